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
