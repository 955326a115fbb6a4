"""The push's chunk and group sizes follow the particle count; they change no
result: every count, from one particle to several chunks per CTA, gives the
bits of the fixed large chunks (apic_set_schedule)."""
import numpy as np
import pytest

from tests.inputs import random_states, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 255, 257, 4099, 120001, 1200001])
def test_push_tiles_change_no_result(prec, n):
    import paper_2307_11107_gb300 as apic
    apic.build()
    cfg = workload(n1=64, n2=32, alpha=0.15, B=1.0, n_init=max(n, 1000), precision=prec, seed=4, sort_interval=2)
    out = []
    for fixed in (False, True):
        s = apic.Sim(cfg)
        if fixed:
            s.set_schedule(chunk_group=4, chunk_items=16)
        for sp, seed, vs in ((0, 11, 1.0), (1, 12, 0.03)):
            s.add_particles(sp, random_states(n, cfg["x1_out"], seed=seed, vscale=vs))
        s.step(3)
        t = s.tallies()
        out.append((s.field("rho"), s.field("phi"), t["bins"], t["counts"], [s.particles(sp) for sp in (0, 1)]))
        s.close()
    (r0, p0, b0, c0, q0), (r1, p1, b1, c1, q1) = out
    assert np.array_equal(r0, r1) and np.array_equal(p0, p1) and np.array_equal(b0, b1) and c0 == c1
    for a, b in zip(q0, q1):
        assert a.shape == b.shape
        assert np.array_equal(a[np.lexsort(a.T[::-1])], b[np.lexsort(b.T[::-1])])


@pytest.mark.parametrize("alpha,grid", [(0.0, (16, 8)), (0.2, (32, 16)), (-0.24, (8, 600))])
def test_fp64_push_at_cell_edges_and_poles(alpha, grid):
    """FP64 particles exactly on grid nodes, on both poles, on the outer
    surface and within rounding of the cell edges, at rest and moving, against
    the oracle: the index-clamped cells, the integer deposit weights and the
    products with reciprocal roots.  Tolerances of the random-state step test
    (test_gpu_parity.py::test_single_step_fp64)."""
    import oracle
    import paper_2307_11107_gb300 as apic
    apic.build()
    n1, n2 = grid
    cfg = workload(n1=n1, n2=n2, alpha=alpha, B=0.7, n_init=5000, precision="fp64", no_inject=True,
                   poisson_tol=1e-13, poisson_max_iter=60)
    x1 = -1.0 + (cfg["x1_out"] + 1.0) / n1 * np.arange(1, n1 + 1)
    x1[-1] = cfg["x1_out"]
    x2 = -1.0 + 2.0 / n2 * np.arange(n2 + 1)
    x1 = np.concatenate([x1, np.nextafter(x1[:-1], 0.0), np.nextafter(x1[:-1], -1.0)])
    x2 = np.concatenate([x2, np.nextafter(x2[:-1], 2.0), np.nextafter(x2[1:], -2.0)])
    if x2.size > 100:
        x2 = x2[:: x2.size // 50]
    x2[:2] = (-1.0, 1.0)
    p = np.stack(np.meshgrid(x1, x2, indexing="ij"), -1).reshape(-1, 2)
    rng = np.random.default_rng(7)
    v = rng.standard_normal((p.shape[0], 3)) * (np.arange(p.shape[0]) % 3 > 0)[:, None]
    s, o = apic.Sim(cfg), oracle.Sim(cfg)
    for sp, vs in ((0, 1.0), (1, 0.03)):
        st = np.column_stack([p, vs * v])
        s.add_particles(sp, st)
        o.add_particles(sp, st)
    s.step(1)
    o.step(1)
    for sp in (0, 1):
        g, r = s.particles(sp), o.particles(sp)[0]
        assert g.shape == r.shape
        assert np.abs(g - r).max() < 1e-9
    # the push's own deposit: the node charges (rho V, each side with its own
    # volumes: their quadratures differ next to a sharp pole) the oracle finds
    # for the positions the GPU holds
    o = oracle.Sim(cfg)
    for sp in (0, 1):
        o.add_particles(sp, s.particles(sp))
    s.step(1)
    o.step(1)
    q, q_o = s.field("rho") * s.field("V"), o.grid("rho") * o.grid("V")
    assert np.abs(q - q_o).max() < 1e-11 * np.abs(q_o).max()
