"""Adjoint of vectors at the ends of the FP32 range: finite products whose sums exceed FLT_MAX (the sums are FP64: finite),
and an infinite element, which may reach only the parameters that move particles out of or into its determinant."""
import itertools

import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def unit(orbits, spe, tb, Z, Nn, twoM, t):
    e = np.zeros(len(spe))
    e[t:t + 1] = 1.0
    o = O.Oracle(orbits, Z, Nn, twoM, 0)
    return o.set_interaction(e, [(*tb[t - len(spe)][:6], 1.0)] if t >= len(spe) else []).matrix()


@pytest.mark.parametrize("name,Z,Nn,twoM", [("sd", 2, 2, 0), ("sd", 3, 4, 1), ("sd", 0, 4, 0)])
def test_sums_beyond_the_fp32_range(name, Z, Nn, twoM):
    """Same tolerance as for any FP32 vectors: (k + 1) 2^-24 sum |gy| |H_t| |x|, at k = 1."""
    orbits, spe, tb = I.space(name)
    c = N.make(orbits, spe, tb, Z, Nn, twoM, +1, device=0)
    g = np.random.default_rng(7)
    x, gy = ((2.0 ** 63 * (1 + 0.4 * g.random((c.dim, 1)))).astype(np.float32) for _ in range(2))
    assert np.all(np.isfinite(x * gy))
    n = len(spe) + len(tb)
    got = c.apply_H_backward(torch.from_numpy(x).cuda(), torch.from_numpy(gy).cuda(), torch.empty((c.dim, 1), device="cuda"),
                             1, N.BS_F32, n_theta=n)
    c.close()
    xh, gh = x.astype(np.float64), gy.astype(np.float64)
    for t in range(0, n, 5):
        H = unit(orbits, spe, tb, Z, Nn, twoM, t)
        tol = 2 * 2.0 ** -24 * np.sum(np.abs(gh) * (abs(H) @ np.abs(xh)))
        assert abs(got[t] - np.sum(gh * (H @ xh))) <= tol, t


def reaches(st, occ, el):
    """Whether element el moves two particles of the determinant occ (proton bits, neutron bits), either way round."""
    a, b, c, d, _, T = el
    inorb = lambda q: [s for s, o in enumerate(st) if o[0] == q - 1]
    for (a, b, c, d) in ((a, b, c, d), (a, b, d, c), (c, d, a, b), (c, d, b, a)):   # a pair's labels have no order
        for x, y in ((0, 1), (1, 0)) + (((0, 0), (1, 1)) if T == 1 else ()):
            for i, j in itertools.product(inorb(a), inorb(b)):
                if not (occ[x] >> i & 1 and occ[y] >> j & 1) or (x == y and i == j):
                    continue
                left = list(occ)
                left[x] &= ~(1 << i)
                left[y] &= ~(1 << j)
                for k, l in itertools.product(inorb(c), inorb(d)):
                    if st[k][1] + st[l][1] != st[i][1] + st[j][1] or (x == y and k == l):
                        continue
                    if not (left[x] >> k & 1 or left[y] >> l & 1):
                        return True
    return False


@pytest.mark.parametrize("Z,Nn,twoM", [(1, 10, 1), (10, 1, 1), (2, 9, 1)])
@pytest.mark.parametrize("k,dtype", [(1, N.BS_F32), (4, N.BS_F32), (1, N.BS_F64)])
@pytest.mark.parametrize("side", [0, 1])
def test_an_infinite_element(Z, Nn, twoM, k, dtype, side):
    orbits, spe, tb = I.space("sd")
    st = [(q, m) for q, o in enumerate(orbits) for m in range(-o.twoj, o.twoj + 1, 2)]
    c = N.make(orbits, spe, tb, Z, Nn, twoM, +1, device=0)
    B = c.export_basis()
    n = len(spe) + len(tb)
    tdt = torch.float64 if dtype == N.BS_F64 else torch.float32
    clean = [torch.from_numpy(I.random_block(c.dim, k, seed=s)).to("cuda", tdt) for s in (3, 4)]
    apart = 0
    for b, (ps, ns, off) in enumerate(B["blocks"]):
        nN = int(B["n_sec"][ns][3])
        d = int(off) + (7 * b) % (int(B["p_sec"][ps][3]) * nN)   # one determinant of every block
        occ = (int(B["p_bits"][B["p_sec"][ps][2] + (d - off) // nN]), int(B["n_bits"][B["n_sec"][ns][2] + (d - off) % nN]))
        v = [q.clone() for q in clean]
        v[side][d] = float("inf")
        got = c.apply_H_backward(v[0], v[1], torch.empty_like(v[0]), k, dtype, n_theta=n)
        v[side][d] = 0.0
        ref = c.apply_H_backward(v[0], v[1], torch.empty_like(v[0]), k, dtype, n_theta=n)
        assert not np.all(np.isfinite(got))
        for t in range(n):
            if t < len(spe):
                hit = any((occ[0] | occ[1]) >> s & 1 for s, o in enumerate(st) if o[0] == t)
            else:
                hit = reaches(st, occ, tb[t - len(spe)][:6])
            if not hit:   # the same terms, in another order: FP64 sums of FP32 or FP64 products
                apart += 1
                assert abs(got[t] - ref[t]) <= (1e-12 if dtype == N.BS_F64 else (k + 1) * 2.0 ** -24) * 256 * k, (d, t)
    assert apart > 0
    c.close()
