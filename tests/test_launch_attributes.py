"""Kernel attributes (shared memory above the default) belong to the device that is
current when they are set: they may not be set once for the process, by the first
context, or a context on another device fails at its first step.  One device
cannot show that, so the source is looked at."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_04605_gb300", "csrc")


def test_attributes_are_not_set_once_for_the_process():
    calls = 0
    for path in glob.glob(os.path.join(CSRC, "*")):
        text = open(path).read()
        for m in re.finditer("cudaFuncSetAttribute", text):
            statement = re.split(r"[;{}]", text[:m.start()])[-1]
            assert "static" not in statement and "call_once" not in statement, (path, statement)
            calls += 1
    assert calls > 0


def test_size_rules_ask_for_the_sm_count():
    """Rules on sites an SM take the count of the device, not that of one chip."""
    for path in glob.glob(os.path.join(CSRC, "*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\b(148|152)\s*\*|\*\s*(148|152)\b", code), path
