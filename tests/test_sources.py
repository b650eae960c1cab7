"""Rules of the CUDA sources that no result shows by itself."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_11102_gb300", "csrc")


def code(name):
    """The text of a source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_reverse_divides_with_correct_rounding():
    """The FP32 reverse takes no approximate reciprocal or division of its own
    (its seeds and weights are quotients whose errors add up over all faces)."""
    assert not re.findall(r"rcp_approx|\bw[n]?rcp\b|__fdividef|rcp\.approx|div\.approx", code("gks_adjoint.cu"))
