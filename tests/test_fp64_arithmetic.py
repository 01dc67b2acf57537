"""What the FP64 kernels may not do with less precision than FP64 rounding gives."""
import os
import re

from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2511_02021_gb300", "csrc")


def test_roots_are_correctly_rounded():
    """K_h is cs^2 l d sqrt(D_T^2 + D_S^2) with IEEE's root, which holds for every argument: a series
    about an approximate reciprocal root is off by an ulp, gives 0 for subnormal arguments and NaN
    for an infinite one."""
    text = {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read()) for f in os.listdir(CSRC)}
    for f, code in text.items():
        assert not re.search(r"\brsqrt|sqrt\.approx|__dsqrt_r[duz]", code), f
    body = text["dycore64.cu"].split("k_diff_edge(Geo64", 1)[1].split("__global__", 1)[0]
    assert re.search(r"(?<!\w)sqrt\(", body)
