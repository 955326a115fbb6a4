"""Host check of the dataflow sweeps' task records
(paper_2307_11107_gb300/csrc/nd_records.cpp): walked on the host in list order
as the GPU walks them, every record stays within the device's limits, comes
after those it waits for, and the sweeps give the factorisation's solution, in
FP32 and FP64, for square, wide and narrow grids with few and many workers."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2307_11107_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("ndr") / "nd_records_check")
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-pthread", "-o", exe,
                           os.path.join(HERE, "native", "nd_records_check.cpp"), os.path.join(CSRC, "nd_factor.cpp"),
                           os.path.join(CSRC, "nd_records.cpp")])
    return exe


@pytest.mark.parametrize("a,b,leaf,units", [((3, 9), (15, 9), 16, 1), ((31, 17), (63, 33), 16, 608),
                                            ((127, 65), (255, 129), 16, 300), ((95, 49), (159, 81), 9, 40),
                                            ((15, 1025), (31, 513), 16, 608), ((511, 257), (255, 9), 16, 608)])
def test_records_give_the_sweeps(checker, a, b, leaf, units):
    out = subprocess.run([checker] + [str(x) for x in (*a, *b, leaf, units)], capture_output=True, text=True,
                         timeout=300).stdout.split()
    assert out[0] == "OK", out
    # the same sums in another order: FP32 and FP64 rounding of dot products of
    # up to about a thousand terms over up to twenty levels
    assert float(out[1]) < 1e-5, out
    assert float(out[2]) < 1e-12, out
