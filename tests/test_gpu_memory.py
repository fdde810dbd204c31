"""bs_load_interaction where the device has room for everything but the pair-core product's tables: it succeeds, and the
products that would use them run by the other kernels.  The shortage is made of an ordinary allocation, sized from the
device's own figures, and given back before any kernel runs."""
import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_load_without_room_for_the_pair_tables():
    orbits, spe, tb = I.space("pf")
    c = N.make(orbits, spe, tb, 6, 2, 0, +1, device=0)
    x = torch.from_numpy(I.random_block(c.dim, 4, seed=3)).to("cuda", torch.float32)
    out = {}

    def products(key):
        for mode in (1, 16):
            y = torch.empty_like(x)
            c.set_kernel(mode)
            c.apply_H(x, y, 4, N.BS_F32)
            c.sync_status()
            out[key, mode] = y
        c.set_kernel(0)

    products("full")
    assert not torch.equal(out["full", 16], out["full", 1])    # mode 16 sums in another order
    optional = sum(c.table(t, np.uint8).nbytes for t in ("pr_items4", "pr_tiles4", "pr_rows4", "pr_store4", "pr_recs"))
    assert optional > 64 << 20
    torch.cuda.synchronize()
    c.build_basis(orbits, 6, 2, 0, +1)                         # the tables go
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    c.load_interaction(spe, tb)
    used = before - torch.cuda.mem_get_info()[0]
    assert used > optional
    c.build_basis(orbits, 6, 2, 0, +1)
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (used - optional // 2), device="cuda", dtype=torch.uint8)
    c.load_interaction(spe, tb)
    del filler
    torch.cuda.empty_cache()
    products("short")
    assert torch.equal(out["short", 1], out["full", 1])
    assert torch.equal(out["short", 16], out["short", 1])      # fell back to the tiled kernel
    c.load_interaction(spe, tb)
    products("again")
    assert torch.equal(out["again", 16], out["full", 16])
    c.close()
