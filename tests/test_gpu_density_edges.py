"""One-body densities: every (f, j) entry of the warp sums that halve their values lane by lane, at each block size, on
sectors narrower and wider than a warp, one particle, an empty species.  Tolerance, derived: a sum of at most dim FP64
products in any order is off by at most (dim + 8) 2^-53 sum |F| |X|, and that sum is at most |F| |X| (2-norms)."""
import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,Z,Nn,twoM", [("sd", 1, 1, 0), ("sd", 0, 3, 3), ("sd", 5, 2, 1), ("sd", 3, 3, 0), ("pf", 2, 1, 1)])
@pytest.mark.parametrize("k", [1, 2, 4, 8])
def test_every_pair_of_columns(name, Z, Nn, twoM, k):
    orbits, spe, tb = I.space(name)
    par = (Z + Nn) * (orbits[0].l % 2) % 2
    c = N.make(orbits, spe, tb, Z, Nn, twoM, 1 - 2 * par, device=0)
    o = O.Oracle(orbits, Z, Nn, twoM, par)
    F, X = (np.asarray(I.random_block(c.dim, k, seed=s), dtype=np.float64).reshape(c.dim, k) for s in (5, 6))
    rho = c.density(torch.from_numpy(F).cuda(), torch.from_numpy(X).cuda(), k, sum(q.twoj + 1 for q in orbits))
    for f in range(k):
        for j in range(k):
            tol = (c.dim + 8) * 2.0 ** -53 * np.linalg.norm(F[:, f]) * np.linalg.norm(X[:, j])
            assert np.max(np.abs(rho[:, :, :, f, j] - o.density(F[:, f], X[:, j]))) <= tol, (f, j)
    c.close()
