"""The benchmark names its roofline by the parts of a round that the library takes: the rule
is written in both places."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _of(path, pattern):
    with open(os.path.join(ROOT, path)) as f:
        found = re.findall(pattern, f.read())
    assert len(found) == 1, (path, pattern, found)
    return found[0]


def test_parts_of_a_round_agree():
    lib = _of("paper_1203_6402_gb300/csrc/round_simt.cu", r"std::max\(1, std::min\((\d+), c\.cap_round / (\d+)\)\)")
    bench = _of("bench.py", r"parts1 = max\(1, min\((\d+), int\(ell \+ 10\.0 \* ell \*\* 0\.5 \+ 64\.0\) // (\d+)\)\)")
    assert lib == bench
