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


def test_every_header_makes_the_library_stale():
    """build() compiles anew when any file that a source includes is newer."""
    from paper_2603_11102_gb300 import build
    included = set()
    for name in os.listdir(CSRC):
        included |= set(re.findall(r'#include "([^"]+)"', code(name)))
    listed = {os.path.basename(h) for h in build.HEADERS}
    assert included and included <= listed


def test_measured_counts_hash_covers_the_double_single_header(tmp_path, monkeypatch):
    """The figures of profiles/ are tied to every header of the kernels they were taken on."""
    import shutil
    import sys
    monkeypatch.syspath_prepend(ROOT)
    sys.modules.pop("bench", None)
    import bench
    now = bench.source_hash("face_flux")
    copy = tmp_path / "paper_2603_11102_gb300" / "csrc"
    shutil.copytree(CSRC, copy)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.source_hash("face_flux") == now
    with open(copy / "gks_ds.cuh", "a") as f:
        f.write("\n")
    assert bench.source_hash("face_flux") != now
