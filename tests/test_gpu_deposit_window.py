"""apic_deposit_static over its paths: one accumulator or several copies, with
and without the shared-memory window of the outermost rows, and grids whose
cell indices leave fewer fraction bits, against the bilinear weighing in FP64."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,n", [(4, 8, 1), (64, 32, 257), (300, 7, 40001), (512, 256, 400000),
                                     (64, 32, 1000003), (33, 600, 2000001), (200000, 1, 30000),
                                     (3, 100000, 300001), (1, 1, 70000)])
def test_deposit_paths_match_fp64_weighing(n1, n2, n):
    import torch
    import paper_2307_11107_gb300 as apic
    from paper_2307_11107_gb300 import _abi
    apic.build()
    L = _abi.load()
    x1_out = -0.07
    rng = np.random.default_rng(n1 + n)
    # most particles near the outer surface, some on nodes and on the borders
    x1 = np.where(rng.random(n) < 0.7, x1_out - 0.05 * rng.random(n), rng.uniform(-1.0, x1_out, n))
    x2 = rng.uniform(-1.0, 1.0, n)
    x1[: n // 50] = -1.0 + (x1_out + 1.0) / n1 * rng.integers(0, n1, n // 50)
    x2[n // 60: n // 40] = -1.0 + 2.0 / n2 * rng.integers(0, n2 + 1, n // 40 - n // 60)
    x1 = np.clip(x1, -1.0, x1_out)
    x2 = np.clip(x2, -1.0, 1.0)
    ref = np.zeros((n1 + 1) * (n2 + 1))
    cnt = np.zeros_like(ref)
    h1, h2 = (x1_out + 1.0) / n1, 2.0 / n2
    u1, u2 = (x1 + 1.0) / h1, (x2 + 1.0) / h2
    i, j = np.clip(np.floor(u1), 0, n1 - 1).astype(int), np.clip(np.floor(u2), 0, n2 - 1).astype(int)
    f1, f2 = np.clip(u1 - i, 0, 1), np.clip(u2 - j, 0, 1)
    for a, wa in ((0, 1 - f1), (1, f1)):
        for b, wb in ((0, 1 - f2), (1, f2)):
            ref += np.bincount((i + a) * (n2 + 1) + j + b, wa * wb, ref.size)
    # the particles that may reach a node: those of the cells around it, and
    # those next to one of these cells' edges, which rounding may put on either side
    for a in (-1, 0, 1, 2):
        for b in (-1, 0, 1, 2):
            m = (i + a >= 0) & (i + a <= n1) & (j + b >= 0) & (j + b <= n2)
            cnt += np.bincount(((i + a) * (n2 + 1) + j + b)[m], minlength=ref.size)
    bad = np.array([[2.0, 0.1], [-1.5, 0.0], [-0.5, 1.5], [np.nan, 0.0], [-0.5, np.nan], [-np.inf, 0.0], [-0.0, 0.2],
                    [np.nextafter(x1_out, 0.0), 0.3], [np.nextafter(-1.0, -2.0), 0.3], [-0.5, np.nextafter(1.0, 2.0)]])
    t = [torch.tensor(np.concatenate([bad[:, c], x, bad[:, c]]), device="cuda") for c, x in ((0, x1), (1, x2))]
    V = torch.ones(ref.size, dtype=torch.float64, device="cuda")
    rho = torch.full_like(V, np.nan)
    grid = _abi.Grid(n1, n2, x1_out)
    total = n + 2 * len(bad)
    s = torch.cuda.current_stream()
    for _ in range(2):
        assert L.apic_deposit_static(C.byref(grid), t[0].data_ptr(), t[1].data_ptr(), total, 1.0, V.data_ptr(),
                                     rho.data_ptr(), C.c_void_p(s.cuda_stream)) == 0
        got = rho.cpu().numpy()
        # every weight is rounded to F = 62 - bits(n) fraction bits; a coordinate
        # resolves its cell fraction to a few 2^-53 of its cell index, in the reference too
        tol = cnt * (2.0 ** -(62 - total.bit_length()) + 4.0 * max(n1, n2) * 2.0 ** -53) + 1e-12 * ref.max()
        assert np.all(np.abs(got - ref) <= tol)
