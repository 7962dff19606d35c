"""Memory that a call clears or fills is used by kernels on the caller's stream,
which need not be ordered behind the legacy one.  The host code, read as
source, uses no call of the legacy stream for it: it goes to the caller's
stream, or to a stream of the library's own that is waited for in the same
function."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16629_gb300", "csrc")


def functions(text):
    """(name, body) of every function defined at the start of a line."""
    for m in re.finditer(r"^[A-Za-z_][^\n;{}=]*?\b(\w+)\([^;{}]*\)\s*\{$", text, flags=re.M):
        yield m.group(1), text[m.end():text.index("\n}", m.end())]


def test_set_up_memory_is_ordered():
    own = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        assert not re.search(r"cudaMemset\(|cudaMemcpy\([^;]*HostToDevice", text), f
        for name, body in functions(text):
            for stream in ("g->cap", "p->cap"):
                # grow_work clears on the stream it is given
                sets = [m.end() for m in re.finditer(rf"(cudaMem\w+Async|grow_work)\([^;]*{stream}\)", body)]
                if sets:
                    assert f"cudaStreamSynchronize({stream})" in body[sets[-1]:], (f, name)
                    own += 1
    assert own >= 4
