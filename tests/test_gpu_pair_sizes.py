"""FP32 products at k = 1, 2 by pairs of cores at the sizes they are chosen for: pf 4p4n (groups of up to 145 neutron cores,
all 16 rows of a tile; sampled rows), and sectors of 1,651 SDs (five pf particles of one species), whose panels hold 32
floats a row.  That the pair-core kernel ran, and not a kernel it falls back to, shows in the last bits: the tiled kernel
sums in another order.  Tolerance as for every FP32 product: n products rounded by 2^-24 each, n up to 10^3, 4e-5 |H| |x|."""
import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I
from tests.test_gpu_hx import _sample_rows, gpu_apply, setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def both(c, x, k):
    out = {}
    try:
        for mode in (16, 1, 0):
            c.set_kernel(mode)
            out[mode] = gpu_apply(c, x, k, N.BS_F32)
            if mode != 1:
                assert np.array_equal(out[mode], gpu_apply(c, x, k, N.BS_F32))
        c.sync_status()
    finally:
        c.set_kernel(0)
    assert not np.array_equal(out[16], out[1])
    return out


@pytest.mark.parametrize("k", [1, 2])
def test_pf_4p4n(k):
    c, o = setup("pf", 4, 4, 0)
    x = I.random_block(o.dim, k, seed=23).astype(np.float32)
    out = both(c, x, k)
    assert np.array_equal(out[0], out[16])   # the untuned rule names it
    x = x.astype(np.float64)
    rows = _sample_rows(o, 4000, 3)
    assert np.all(np.abs(out[16][rows] - o.apply_rows(rows, x)) <= 4e-5 * o.apply_rows(rows, np.abs(x), absval=True) + 1e-30)
    assert np.all(np.isfinite(out[16]))


@pytest.mark.parametrize("Z,Nn,k", [(1, 5, 1), (5, 1, 1), (5, 1, 2)])   # (1p5n, k = 2: a proton core's rows exceed the kernel's)
def test_narrow_panels(Z, Nn, k):
    c, o = setup("pf", Z, Nn, 0)
    x = I.random_block(o.dim, k, seed=29).astype(np.float32)
    y = both(c, x, k)[16]
    x = x.astype(np.float64)
    rows = _sample_rows(o, 3000, 5)
    assert np.all(np.abs(y[rows] - o.apply_rows(rows, x)) <= 4e-5 * o.apply_rows(rows, np.abs(x), absval=True) + 1e-30)
    assert np.all(np.isfinite(y))
