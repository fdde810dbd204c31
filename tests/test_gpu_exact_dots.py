"""bs_block_dots of FP32 vectors against exactly rounded sums, at the edges of
its tiles (fewer rows than one tile, a ragged last tile, several tiles per
CTA) and with heavy cancellation.  Tolerance from the arithmetic: products
are exact, and every addition into a double-float sum is off by at most
2^-46 of the running sum, itself at most S = sum |v w|; a chain has at most
n <= 25 tiles x 8 rows additions, then 13 joins of partial sums: (n + 13)
2^-46 S, n = rows here at most 200 per thread."""
import math

import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,Z,Nn", [("sd", 1, 1), ("sd", 2, 2), ("sd", 4, 4), ("pf", 3, 3)])
@pytest.mark.parametrize("k,nb", [(1, 2), (2, 3), (4, 1), (8, 3)])
def test_exact_products(name, Z, Nn, k, nb):
    orbits, spe, tb = I.space(name)
    c = N.make(orbits, spe, tb, Z, Nn, 0, +1, device=0)
    dim = c.dim
    g = np.random.default_rng(11 * k + nb)
    V = (g.standard_normal((nb, dim, k)) * 2.0 ** g.integers(-12, 12, (nb, dim, k))).astype(np.float32)
    W = (g.standard_normal((dim, k)) * 2.0 ** g.integers(-12, 12, (dim, k))).astype(np.float32)
    half = dim // 2   # the second half cancels the first but for one part in 2^20
    V[:, half:2 * half] = V[:, :half]
    W[half:2 * half] = -W[:half] * np.float32(1 + 2.0 ** -20)
    C = torch.full((nb * k * k,), float("nan"), device="cuda", dtype=torch.float64)
    c.block_dots(torch.from_numpy(V).cuda(), nb, torch.from_numpy(W).cuda(), k, N.BS_F32, C)
    got = C.cpu().numpy().reshape(nb, k, k)
    c.sync_status()
    c.close()
    for b in range(nb):
        for i in range(k):
            for j in range(0, k, max(1, k // 2)):
                p = V[b, :, i].astype(np.float64) * W[:, j].astype(np.float64)   # exact in 53 bits
                tol = 213 * 2.0 ** -46 * np.sum(np.abs(p)) + 1e-300
                assert abs(got[b, i, j] - math.fsum(p)) <= tol, (b, i, j)
