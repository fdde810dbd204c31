"""Gradients on a context whose basis was rebuilt, with the same element labels, equal those of a fresh context: the
derivative list indexes the tables of the basis it was made for.  A fresh context differs only in the order of FP64
additions (atomics): at most 10^6 2^-53 of sum |terms|; with columns normalized and elements of 2 (2j + 1)^2 <= 128 terms
of magnitude <= 2 that sum is below 256 k."""
import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

J72, J52, J32 = I.Orbit(0, 3, 7), I.Orbit(0, 3, 5), I.Orbit(1, 1, 3)
TB = [(1, 1, 1, 1, 0, 1, -1.5), (1, 1, 1, 1, 2, 1, 0.5), (1, 1, 1, 1, 1, 0, 0.75), (1, 1, 1, 1, 3, 0, -0.25)]


def gradient(c, k, dtype):
    tdt = torch.float64 if dtype == N.BS_F64 else torch.float32
    x, gy = (torch.from_numpy(I.random_block(c.dim, k, seed=s)).to("cuda", tdt) for s in (3, 4))
    return c.apply_H_backward(x, gy, torch.empty_like(gy), k, dtype, n_theta=c.n_spe + c.n_tbme)


@pytest.mark.parametrize("first,second", [([J72], [J52]), ([J52], [J72]), ([J72, J32], [J32, J72])])
@pytest.mark.parametrize("k,dtype", [(1, N.BS_F64), (4, N.BS_F32)])
def test_same_labels_on_another_basis(first, second, k, dtype):
    spe, tb = [0.5, -0.25][:len(first)], TB if len(first) == 1 else TB[:3]
    c = N.make(first, spe, tb, 2, 2, 0, +1, device=0)
    gradient(c, k, dtype)
    c.build_basis(second, 2, 2, 0, +1).load_interaction(spe, tb)
    got = gradient(c, k, dtype)
    f = N.make(second, spe, tb, 2, 2, 0, +1, device=0)
    ref = gradient(f, k, dtype)
    assert np.max(np.abs(got - ref)) <= 1e6 * 2.0 ** -53 * 256 * k
    assert np.max(np.abs(ref)) > 1e-3
    # back on the first basis, then another interaction of the same labels
    c.build_basis(first, 2, 2, 0, +1).load_interaction(spe, [(*t[:6], 2 * t[6]) for t in tb])
    f2 = N.make(first, spe, tb, 2, 2, 0, +1, device=0)
    assert np.max(np.abs(gradient(c, k, dtype) - gradient(f2, k, dtype))) <= 1e6 * 2.0 ** -53 * 256 * k
    for q in (c, f, f2):
        q.close()
