"""The reverse sweep's kernels where they branch: one and several copies of the
gradient adjoint, the transposed solve as dataflow sweeps and level by level,
batches of uneven grids, and particles on nodes, on the axis, on the outermost
row and at rest, against the forward tangents of the same window (FP64)."""
import numpy as np
import pytest

from tests.inputs import random_states, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def apic():
    import paper_2307_11107_gb300 as apic
    apic.build()
    return apic


def _on_edges(st, n1, n2, x1_out):
    """Every 16th particle moved: onto an x2 node, the axis (at rest and
    moving), an x1 node, the outermost row, both."""
    h1 = (x1_out + 1.0) / n1
    st = st.copy()
    q = st[::16]
    kind = np.arange(len(q)) % 6
    q[kind == 0, 1] = -1.0 + (2.0 / n2) * np.rint((q[kind == 0, 1] + 1.0) * n2 / 2.0)
    q[kind == 1, 1] = 1.0
    q[kind == 2, 1] = -1.0
    q[kind == 2, 2:] = 0.0
    q[kind == 3, 0] = -1.0 + h1 * np.clip(np.rint((q[kind == 3, 0] + 1.0) / h1), 2, n1 - 1)
    q[kind == 4, 0] = x1_out
    q[kind == 5, 0] = x1_out
    q[kind == 5, 1] = 0.0
    st[::16] = q
    return st


@pytest.mark.parametrize("flow", ["1", "0"])
@pytest.mark.parametrize("grids,n", [(((32, 16),), 160), (((32, 16), (48, 40)), 9000), (((16, 64), (96, 32)), 3000)])
def test_reverse_sweep_against_forward_tangents(apic, monkeypatch, grids, n, flow):
    monkeypatch.setenv("APIC_ND_FLOW", flow)
    K = 3
    cfgs = [workload(n1=a, n2=b, alpha=0.12 - 0.2 * k, B=0.6, n_init=n, seed=9, instance=k, poisson_tol=1e-13,
                     poisson_max_iter=80) for k, (a, b) in enumerate(grids)]

    def sim():
        s = apic.Sim(cfgs, precision="fp64")
        for k, (a, b) in enumerate(grids):
            for sp in (0, 1):
                st = random_states(n, cfgs[k]["x1_out"], seed=71 + 2 * k + sp, vscale=1.0 if sp == 0 else 0.03)
                s.add_particles(sp, _on_edges(st, a, b, cfgs[k]["x1_out"]), instance=k)
        return s

    s = sim()
    out = s.sensitivity(K)
    s.close()
    w = np.random.default_rng(4).standard_normal((len(grids), 5))
    s = sim()
    g, v = s.adjoint(K, w, values=True)
    s.close()
    for k in range(len(grids)):
        J = out["jacobian"][k]
        # rounding, the solves' tolerance times a condition of some thousands: as the windows' other comparisons
        assert np.all(np.abs(g[k] - w[k] @ J) <= 1e-10 * np.abs(w[k][:, None] * J).sum(axis=0)), (g[k], w[k] @ J)
        assert np.allclose(v[k], out["values"][k], rtol=1e-12, atol=1e-14)
