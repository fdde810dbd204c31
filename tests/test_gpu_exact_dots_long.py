"""bs_block_dots of FP32 vectors over long sums (pf 5p5n, dim 18,600,516, a multiple of four: the streamed kernel at every
k, up to 239 tiles of eight rows a thread), equal products, where rounding errors add up in one direction, and squares of
random numbers.
Tolerance from the arithmetic, u = 2^-24, S = sum |v w|: inside a tile the step j of 8 adds an exact remainder rounded to u
of itself (at most u S) to a sum of remainders of at most j u S, rounded to u of itself: 8 + 36 units of u^2 S for the
tile's share; every joining of two normalized pairs (the tiles of a thread, 5 lane steps, 8 warps) rounds remainders of at
most 3 u S twice: 6 u^2 S each.  The sums over CTAs are FP64: 304 x 2^-53 S, below one unit more."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_ctx = []


def context():
    if not _ctx:
        orbits, spe, tb = I.space("pf")
        _ctx.append(N.make(orbits, spe, tb, 5, 5, 0, +1, device=0))
    return _ctx[0]


def tolerance(dim, k):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-(-(-dim * k // 2048)) // (2 * nsm))
    return (44 + 6 * (tiles + 13) + 1) * 2.0 ** -48


def dots(c, V, W, k):
    C = torch.full((V.shape[0] * k * k,), float("nan"), device="cuda", dtype=torch.float64)
    c.block_dots(V, V.shape[0], W, k, N.BS_F32, C)
    c.sync_status()
    return C.cpu().numpy().reshape(V.shape[0], k, k)


@pytest.mark.parametrize("k", [1, 2, 4, 8])
def test_equal_products(k):
    c = context()
    g = np.random.default_rng(5)
    a, b = ((1 + g.random((n, k))).astype(np.float32) for n in (2, 1))
    V = torch.from_numpy(a).cuda()[:, None, :].expand(2, c.dim, k).contiguous()
    W = torch.from_numpy(b).cuda().expand(c.dim, k).contiguous()
    got = dots(c, V, W, k)
    for n in range(2):
        for i in range(k):
            for j in range(k):
                ref = c.dim * Fraction(float(a[n, i])) * Fraction(float(b[0, j]))
                assert abs(Fraction(float(got[n, i, j])) - ref) <= Fraction(tolerance(c.dim, k)) * ref, (n, i, j)


@pytest.mark.parametrize("k", [1, 8])
def test_squares(k):
    c = context()
    V = torch.randn((1, c.dim, k), device="cuda", generator=torch.Generator(device="cuda").manual_seed(k))
    got = dots(c, V, V[0].contiguous(), k)
    h = V[0].double().cpu().numpy()
    for i in range(0, k, 3):
        ref = math.fsum(h[:, i] * h[:, i])   # the products are exact in 53 bits
        assert abs(got[0, i, i] - ref) <= tolerance(c.dim, k) * ref, i
