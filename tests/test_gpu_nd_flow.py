"""The nested-dissection dataflow solve with FP64 fronts (FP64 particles)
against the oracle's banded LU, on grids from a few fronts to several thousand,
square, wide and narrow; a tolerance below FP64 rounding ends at the rounding
floor; and the FP32 sweeps give the level-by-level sweeps' bits."""
import numpy as np
import pytest

import oracle
from tests.inputs import random_rho, workload

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("n1,n2", [(4, 8), (8, 16), (40, 24), (64, 300), (16, 1024), (300, 28), (288, 144)])
@pytest.mark.parametrize("tol", [1e-12, 1e-17])
def test_fp64_fronts_match_banded_lu(n1, n2, tol):
    """Tolerance as test_gpu_parity.py::test_poisson_fp64_matches_banded_lu."""
    import paper_2307_11107_gb300 as apic
    apic.build()
    cfg = workload(n1=n1, n2=n2, alpha=0.2, x1_out=-0.05, n_init=1000, precision="fp64", poisson_tol=tol,
                   poisson_max_iter=30)
    rho = random_rho(n1, n2, seed=n1 + n2, scale=0.3)
    s, o = apic.Sim(cfg), oracle.Sim(cfg)
    assert s.stats()["solver"].startswith("FP64 nested dissection")
    assert rel(s.solve_poisson(rho), o.solve(rho)) < 1e-10
    s.close()


@pytest.mark.parametrize("grids", [[(32, 32)], [(96, 200)], [(128, 64), (256, 128), (96, 48), (16, 300)]])
def test_fp32_dataflow_gives_the_level_by_level_bits(grids, monkeypatch):
    import paper_2307_11107_gb300 as apic
    apic.build()
    monkeypatch.setenv("APIC_DIRECT", "nd")
    cfgs = [workload(n1=a, n2=b, alpha=0.15, x1_out=-0.05, n_init=1000, precision="fp32", poisson_tol=1e-4,
                     poisson_max_iter=30, instance=k) for k, (a, b) in enumerate(grids)]
    out = []
    for flow in ("1", "0"):
        monkeypatch.setenv("APIC_ND_FLOW", flow)
        s = apic.Sim(cfgs)
        out.append([s.solve_poisson(random_rho(a, b, seed=5 + k, scale=0.3), instance=k)
                    for k, (a, b) in enumerate(grids)])
        s.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
