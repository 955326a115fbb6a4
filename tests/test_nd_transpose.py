"""Host check of the reverse sweep's transposed solve: the records of the
transposed fronts (paper_2307_11107_gb300/csrc/nd_records.cpp), walked as the
GPU walks them, give A^-T: y . A^-1 r = (A^-T y) . r."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2307_11107_gb300", "csrc")


@pytest.mark.parametrize("a,b,units", [((3, 9), (15, 9), 1), ((31, 17), (63, 33), 608), ((255, 129), (40, 90), 300),
                                       ((9, 201), (255, 9), 40)])
def test_transposed_records(tmp_path, a, b, units):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "check")
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-pthread", "-o", exe,
                           os.path.join(HERE, "native", "nd_transpose_check.cpp"),
                           os.path.join(CSRC, "nd_factor.cpp"), os.path.join(CSRC, "nd_records.cpp")])
    out = subprocess.run([exe] + [str(x) for x in (*a, *b, units)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out
    # FP64 rounding of dot products over up to twenty tree levels
    assert float(out.stdout.split()[1]) < 1e-13, out.stdout
