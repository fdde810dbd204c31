"""The adjoint's double-float sums by themselves: FP32 vectors whose products are exact in FP32 (11-bit mantissas over 13
binary orders, one nonzero column per state, so that a k-term product is one product), so that only the sums can be off.
Units with many columns: neutron cores (pf 1p5n), neutron SDs under two protons (sd 2p6n).
Tolerance per parameter, u = 2^-24, S = sum |gy| |H_t| |x|: the sums are normalized after at most 15 additions, the j-th of
which rounds a remainder of at most u S and their sum, at most j u S, to u of themselves: 135 u^2 S, at most ncol / 8 + 1
times.  At most 256 slices' sums meet: two roundings each of remainders of at most 25 u S.  FP64 collects at most 10^6
units' sums.  (Plain FP32 sums would be off by about 2^-24 S.)"""
import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def exact_block(dim, k, seed):
    g = np.random.default_rng(seed)
    v = g.integers(-2047, 2048, dim) * 2.0 ** g.integers(-6, 7, dim)
    x = np.zeros((dim, k), dtype=np.float32)
    x[np.arange(dim), np.random.default_rng(99).integers(0, k, dim)] = v
    return x


@pytest.mark.parametrize("name,Z,Nn,ncol", [("pf", 1, 5, 500), ("sd", 2, 6, 142)])
def test_sums_of_exact_products(name, Z, Nn, ncol):
    orbits, spe, tb = I.space(name)
    c = N.make(orbits, spe, tb, Z, Nn, 0, +1, device=0)
    n = len(spe) + len(tb)
    some = range(0, n, 1 + n // 8)
    H = {}
    for t in some:
        e = np.zeros(len(spe))
        e[t:t + 1] = 1.0
        o = O.Oracle(orbits, Z, Nn, 0, 0)
        H[t] = o.set_interaction(e, [(*tb[t - len(spe)][:6], 1.0)] if t >= len(spe) else []).matrix()
    for k in (1, 2, 4, 8):
        x, gy = exact_block(c.dim, k, 3 + k), exact_block(c.dim, k, 30 + k)
        g = c.apply_H_backward(torch.from_numpy(x).cuda(), torch.from_numpy(gy).cuda(), torch.empty((c.dim, k), device="cuda"),
                               k, N.BS_F32, n_theta=n)
        x, gy = x.astype(np.float64), gy.astype(np.float64)
        for t in some:
            rel = (135 * (ncol // 8 + 1) + 50 * 256) * 2.0 ** -48 + 1e6 * 2.0 ** -53
            tol = rel * np.sum(np.abs(gy) * (abs(H[t]) @ np.abs(x)))
            assert abs(g[t] - np.sum(gy * (H[t] @ x))) <= tol, (k, t)
    c.close()
