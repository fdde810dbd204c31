"""bs_lanczos where the device has too little memory: BS_ENOMEM and a usable context, nothing launched without its buffers.
(The basis asked for is larger than the whole device, so the call cannot succeed.)"""
import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def context():
    orbits, spe, tb = I.space("pf")
    return N.make(orbits, spe, tb, 4, 4, 0, +1, device=0)


@pytest.mark.parametrize("use_graph", [False, True])
def test_a_basis_larger_than_the_device(use_graph):
    c = context()
    total = torch.cuda.mem_get_info()[1]
    niter = 40000
    assert (niter + 1) * c.dim * 4 > total
    x = torch.randn((c.dim, 1), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    y, y2 = torch.empty_like(x), torch.empty_like(x)
    c.apply_H(x, y, 1, N.BS_F32)
    with pytest.raises(N.BSError) as e:
        c.lanczos(x, 1, N.BS_F32, niter, 1, refine=False, use_graph=use_graph)
    assert "ENOMEM" in str(e.value)
    c.apply_H(x, y2, 1, N.BS_F32)
    torch.cuda.synchronize()
    assert torch.equal(y, y2)
    ev, rep = c.lanczos(x, 1, N.BS_F32, 10, 1, refine=False, use_graph=use_graph)
    assert np.all(np.isfinite(ev)) and rep["iterations"] == 10
    c.close()


def test_the_stored_basis_comes_before_the_workspace():
    """FP32 k = 2: the products' workspace (Z = 4 partial vectors, 63 MB) does not fit beside the stored basis, the basis
    alone does: the run succeeds (on a kernel without workspace) with the levels of an unhindered one, to the rounding of
    FP32 products (4e-5 |H| |x| per element; ten levels' worth of iterations stay within 1e-3 of |E|)."""
    c = context()
    k, niter = 2, 12
    x = torch.from_numpy(I.random_block(c.dim, k, seed=3)).to("cuda", torch.float32)
    y = torch.empty_like(x)
    c.set_kernel(2)
    c.apply_H(x, y, k, N.BS_F32)                     # the row kernel is loaded
    c.set_kernel(0)
    ev, _ = c.lanczos(x, k, N.BS_F32, niter, 2, refine=False)
    c.close()
    c = context()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    block, part = c.dim * k * 4, 4 * c.dim * k * 4
    need = (niter + 2) * block
    filler = torch.empty(torch.cuda.mem_get_info()[0] - need - part // 2, device="cuda", dtype=torch.uint8)
    got, rep = c.lanczos(x, k, N.BS_F32, niter, 2, refine=False)
    del filler
    torch.cuda.empty_cache()
    assert rep["iterations"] == niter
    assert np.max(np.abs(got - ev)) <= 1e-3 * np.max(np.abs(ev))
    again, _ = c.lanczos(x, k, N.BS_F32, niter, 2, refine=False)
    assert np.array_equal(again, ev)
    c.close()
