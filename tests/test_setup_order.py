"""Memory that a call clears or fills by the legacy stream is used by kernels on
the caller's stream, which need not be ordered behind that one: the host code,
read as source, waits for the legacy stream in the function that does it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16629_gb300", "csrc")
LEGACY = r"cudaMemset\(|cudaMemcpy\([^;]*HostToDevice"


def functions(text):
    """(name, body) of every function defined at the start of a line."""
    for m in re.finditer(r"^[A-Za-z_][^\n;{}=]*?\b(\w+)\([^;{}]*\)\s*\{$", text, flags=re.M):
        yield m.group(1), text[m.end():text.index("\n}", m.end())]


def test_legacy_stream_work_is_waited_for():
    bodies = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            with open(os.path.join(CSRC, f)) as fh:
                bodies.update(functions(re.sub(r"//[^\n]*", "", fh.read())))
    setters = {n: b for n, b in bodies.items() if re.search(LEGACY, b)}
    assert {"alloc_base", "shift_tc_reserve", "act_grid_create", "act_grid_status", "ragged_build"} <= set(setters)
    for n, body in setters.items():
        assert "settle()" in body[[m.end() for m in re.finditer(LEGACY, body)][-1]:], n
