"""The fields and gradients are formed with rounded operations.  The approximate
intrinsics stand in one place, where they always were: the acoustic pass on rows of
whole 16-byte units divides by 1 + sd with one."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_10519_gb300", "csrc")
APPROXIMATE = r"__fdividef|__frsqrt_rn|__expf|__logf|__sinf|__cosf|__powf|__saturatef|\w+\.approx\w*"


def test_where_approximate_intrinsics_stand():
    found = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        with open(f) as src:
            hits = re.findall(APPROXIMATE, re.sub(r"//[^\n]*", "", src.read()))
        if hits:
            found[os.path.basename(f)] = hits
    assert found == {"stencil_tma.cu": ["__fdividef"] * 2}, found


def test_no_flag_makes_operations_approximate():
    from paper_2004_10519_gb300 import _build
    assert not any(w in f for f in _build.NVCC_FLAGS for w in ("fast_math", "prec-div", "prec-sqrt", "ftz"))
