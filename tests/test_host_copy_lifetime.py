"""An asynchronous copy out of a call's own pageable memory has to be over
before that memory goes: the functions of the library's host code, read as
source, wait for their stream behind every such copy."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16629_gb300", "csrc")


def test_copies_from_local_vectors_are_waited_for():
    checked = 0
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"cudaMemcpyAsync\([^;]*?(\w+)\.data\(\)[^;]*;", text):
            function = text[m.end():text.index("\n}", m.end())]
            wait = function.find("cudaStreamSynchronize")
            # nothing but the error check of the copy itself in front of it
            assert wait >= 0 and ";" not in function[:wait], (f, m.group(0))
            checked += 1
    assert checked >= 1
