"""Kernels launched as programmatic dependents, read as source (no GPU).

Such a kernel may start while the kernel before it still runs.  What earlier
kernels of a decomposition write is visible to it only behind its own
griddepcontrol.wait, so in front of that wait it may use pointers only to what
is constant since the dictionary's build."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16629_gb300", "csrc")
WAIT = "griddepcontrol.wait"
# written by the dictionary's build and by nothing after it
CONSTANT = {"D", "D32", "tpl", "scale", "scaleT", "span", "blk_order", "eps_bits"}
# (kernel, pointer) used in front of the wait for a reason given there
BEFORE = {
    # the samples do not depend on the residual, and what used them before is
    # complete when the update lets this kernel start; it waits at its end
    ("k_lem_lhs", "cand"), ("k_lem_lhs", "ncand"),
}


def _closing(text, i):
    depth = 0
    for k in range(i, len(text)):
        depth += {"(": 1, "{": 1, ")": -1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def _strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def kernels():
    """(name, {pointer parameter: its declaration}, body) of every kernel that waits."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = _strip_comments(fh.read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            close = _closing(text, m.end() - 1)
            start = text.index("{", close)
            body = text[start:_closing(text, start)]
            if WAIT not in body:
                continue
            pointers = {}
            for p in text[m.end():close].split(","):
                if "*" in p:
                    pointers[re.search(r"(\w+)\s*$", p).group(1)] = " ".join(p.split())
            out.append((m.group(1), pointers, body))
    return out


KERNELS = kernels()


def test_the_kernels_are_found():
    names = {name for name, _, _ in KERNELS}
    assert {"k_gemv", "k_gemv_stream", "k_gemv_multi", "k_update", "k_update_refined", "k_rescan", "k_shift_rows",
            "k_shift_gemm", "k_shift_flag", "k_shift_rescan", "k_shift_search", "k_shift_update", "k_lem_lhs",
            "k_lem_screen", "k_lem_pick"} <= names


@pytest.mark.parametrize("name,pointers,body", KERNELS, ids=[k[0] for k in KERNELS])
def test_nothing_earlier_kernels_write_is_used_before_the_wait(name, pointers, body):
    before = body[:body.index(WAIT)]
    for p in pointers:
        if p in CONSTANT or (name, p) in BEFORE:
            continue
        assert not re.search(rf"\b{p}\b", before), f"{name} uses {p} before it waits"
    if name == "k_shift_search":  # its pointers come in a struct; what selects the form is its own argument
        used = set(re.findall(r"\bA\.(R|keys|scores|chlist|count_dev|status)\b", before))
        assert used <= {"count_dev"} and "*A.count_dev" not in before


@pytest.mark.parametrize("name,pointers,body", KERNELS, ids=[k[0] for k in KERNELS])
def test_only_constants_are_restrict(name, pointers, body):
    """An access through a __restrict__ pointer may be moved ahead of the
    wait (the compiler has done so with a queue's length)."""
    assert [p for p, decl in pointers.items() if "__restrict__" in decl and p not in CONSTANT] == []
