"""What the kernels' sources have to keep to, checked on the text (no GPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_3631_gb300", "csrc")


def arguments(text, call):
    """The argument texts of every `call(...)` in text."""
    for m in re.finditer(r"\b%s\s*\(" % call, text):
        depth, k = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        yield text[m.end():k - 1]


def test_non_coherent_loads_address_constant_tables_only():
    # __ldg promises memory that nothing writes while the kernel runs; a step's blocks are
    # resident while the previous step still writes the state or co-state they will read
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        assert "ld.global.nc" not in text, path
        for arg in arguments(text, "__ldg"):
            seen += 1
            assert not re.search(r"\b(lin|lout|buf|wave|gbar|ring)\b", arg), (path, arg)
    assert seen
