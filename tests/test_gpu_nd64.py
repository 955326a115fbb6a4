"""FP64 nested-dissection fronts under FP32 particles (the default on small grids
with a tight tolerance; APIC_DIRECT=nd64): the same fields as FP32 fronts give,
alone and batched, and the rule that chooses them."""
import numpy as np
import pytest

from tests.inputs import random_rho, random_states, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def apic():
    import paper_2307_11107_gb300 as apic
    apic.build()
    return apic


@pytest.mark.parametrize("grids", [((16, 8),), ((160, 80),), ((96, 200),), ((40, 24), (264, 92))])
def test_fp64_fronts_give_the_same_fields(apic, monkeypatch, grids):
    out = {}
    for mode in ("nd", "nd64"):
        monkeypatch.setenv("APIC_DIRECT", mode)
        cfgs = [workload(n1=a, n2=b, alpha=0.15, B=0.5, n_init=4000, seed=3, instance=k, poisson_tol=1e-11,
                         poisson_max_iter=30) for k, (a, b) in enumerate(grids)]
        s = apic.Sim(cfgs, precision="fp32")
        assert s.stats()["solver"].startswith("FP64" if mode == "nd64" else "FP32")
        for k in range(len(grids)):
            for sp in (0, 1):
                s.add_particles(sp, random_states(4000, cfgs[k]["x1_out"], seed=5 + sp, vscale=1.0 if sp == 0 else 0.03),
                                instance=k)
        s.step(1)
        r = []
        for k, (a, b) in enumerate(grids):
            r += [s.field("phi", k), s.field("G1", k), s.field("G2", k), s.solve_poisson(random_rho(a, b, 7), instance=k)]
        out[mode] = r
        s.close()
    for q, (x, y) in enumerate(zip(out["nd"], out["nd64"])):
        # the tolerance times the condition of the solved operator (some hundreds); the gradients are FP32 values
        tol = 1e-6 if q % 4 in (1, 2) else 1e-8
        assert np.abs(x - y).max() <= tol * np.abs(x).max(), q


@pytest.mark.parametrize("n1,n2,tol,want", [(256, 128, 1e-10, "FP64 nested"), (256, 128, 1e-8, "FP32 nested"),
                                            (512, 256, 1e-10, "FP32 nested"), (64, 32, 1e-10, "FP32 block")])
def test_which_fronts(apic, monkeypatch, n1, n2, tol, want):
    monkeypatch.delenv("APIC_DIRECT", raising=False)
    s = apic.Sim(workload(n1=n1, n2=n2, alpha=0.15, n_init=1000, poisson_tol=tol), precision="fp32")
    assert s.stats()["solver"].startswith(want)
    s.close()
