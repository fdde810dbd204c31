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
