"""Gram-matrix densities of the adjoint at the edges of their range: species with no, one or two particles (no pn term,
no like-particle cores), nearly filled shells, odd and negative-parity spaces, every block size, against the oracle's
unit-parameter matrices.  Tolerance per parameter, derived from the arithmetic: FP32 vectors form each k-term product sum
in FP32 (k roundings of 2^-24), all else carries 48 bits or more, so |error| <= (k + 1) 2^-24 sum |gy| |H_t| |x|; FP64 sums
of up to 10^6 terms, 10^6 2^-53 of the same sum."""
import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPACES = [("sd", 1, 1, 0), ("sd", 2, 0, 0), ("sd", 0, 3, 3), ("sd", 3, 1, 2), ("sd", 11, 2, 1), ("p", 3, 3, 0), ("pf", 2, 1, 1)]


@pytest.mark.parametrize("name,Z,Nn,twoM", SPACES)
@pytest.mark.parametrize("k,dtype", [(1, N.BS_F32), (2, N.BS_F32), (8, N.BS_F32), (1, N.BS_F64), (4, N.BS_F64), (8, N.BS_F64)])
def test_every_parameter(name, Z, Nn, twoM, k, dtype):
    orbits, spe, tb = I.space(name)
    par = (Z + Nn) * (orbits[0].l % 2) % 2
    c = N.make(orbits, spe, tb, Z, Nn, twoM, 1 - 2 * par, device=0)
    tdt = torch.float64 if dtype == N.BS_F64 else torch.float32
    x, gy = (torch.from_numpy(I.random_block(c.dim, k, seed=s)).to("cuda", tdt) for s in (3, 4))
    gx = torch.empty_like(gy)
    n = len(spe) + len(tb)
    g = c.apply_H_backward(x, gy, gx, k, dtype, n_theta=n)
    again = c.apply_H_backward(x, gy, gx, k, dtype, n_theta=n)
    c.close()
    xh, gh = x.double().cpu().numpy(), gy.double().cpu().numpy()
    o = O.Oracle(orbits, Z, Nn, twoM, par)
    rel = (k + 1) * 2.0 ** -24 if dtype == N.BS_F32 else 1e6 * 2.0 ** -53
    for t in range(n):
        e = np.zeros(len(spe))
        unit = []
        if t < len(spe):
            e[t] = 1.0
        else:
            unit = [(*tb[t - len(spe)][:6], 1.0)]
        H = o.set_interaction(e, unit).matrix()
        tol = rel * np.sum(np.abs(gh) * (abs(H) @ np.abs(xh))) + 1e-300
        assert abs(g[t] - np.sum(gh * (H @ xh))) <= tol, t
        assert abs(again[t] - g[t]) <= tol, t
