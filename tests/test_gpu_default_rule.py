"""Which kernel the default mode runs, shown by its last bits (every kernel sums in its own order): the sizes at which a
neighbouring kernel of the rule takes a sixth to two thirds longer.  FP64: wide sectors over a full chip of rows keep the
pipelined kernel below 50,000 states.  FP32: 190 rows of 565 columns (86,810 states) keep the core-grouped kernel; 20 proton
cores are too few for pairs of cores at k = 1, and 190 at k = 4."""
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_ctx = {}


@pytest.mark.parametrize("name,Z,Nn,dtype,k,mode,other", [
    ("sd", 3, 6, N.BS_F64, 2, 6, 1), ("sd", 3, 5, N.BS_F64, 4, 6, 1), ("pf", 2, 3, N.BS_F64, 8, 6, 1),
    ("sd", 4, 4, N.BS_F64, 2, 1, 6), ("sd", 4, 4, N.BS_F64, 1, 1, 2),
    ("pf", 2, 4, N.BS_F32, 4, 20, 1), ("pf", 2, 4, N.BS_F32, 8, 20, 1), ("pf", 2, 4, N.BS_F32, 1, 1, 16),
    ("pf", 2, 5, N.BS_F32, 1, 2, 16), ("pf", 3, 4, N.BS_F32, 4, 20, 16), ("pf", 3, 4, N.BS_F32, 1, 16, 2),
    ("sd", 4, 4, N.BS_F32, 4, 1, 16)])
def test_default_kernel(name, Z, Nn, dtype, k, mode, other):
    if (name, Z, Nn) not in _ctx:
        orbits, spe, tb = I.space(name)
        par = (-1) ** ((Z + Nn) * (orbits[0].l % 2) % 2)
        _ctx[name, Z, Nn] = N.make(orbits, spe, tb, Z, Nn, (Z + Nn) % 2, par, device=0)
    c = _ctx[name, Z, Nn]
    x = torch.from_numpy(I.random_block(c.dim, k, seed=9)).to("cuda", torch.float64 if dtype == N.BS_F64 else torch.float32)
    y = {}
    for m in (0, mode, other):
        c.set_kernel(m)
        y[m] = torch.empty_like(x)
        c.apply_H(x, y[m], k, dtype)
    c.set_kernel(0)
    c.sync_status()
    assert torch.equal(y[0], y[mode])
    assert not torch.equal(y[mode], y[other])
