"""A product captured in a CUDA graph stays replayable when later calls need a larger workspace: the graph's own
workspace is neither freed nor handed to anyone else.  Bit-identical results; the memory allocated after the larger
call, where a freed workspace would be found again, keeps its pattern."""
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,mode", [(1, 16), (2, 16), (4, 16), (4, 20)])
def test_replay_after_a_larger_workspace(k, mode):
    orbits, spe, tb = I.space("sd")
    c = N.make(orbits, spe, tb, 5, 6, 1, +1, device=0)
    x = torch.from_numpy(I.random_block(c.dim, k, seed=5)).to("cuda", torch.float32)
    y, ref = torch.empty_like(x), torch.empty_like(x)
    c.set_kernel(mode)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        c.apply_H(x, ref, k, N.BS_F32, st.cuda_stream)
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        c.apply_H(x, y, k, N.BS_F32, st.cuda_stream)
    x8 = torch.from_numpy(I.random_block(c.dim, 8, seed=6)).to("cuda", torch.float32)
    y8 = torch.empty_like(x8)
    c.apply_H(x8, y8, 8, N.BS_F32)                      # the workspace grows
    torch.cuda.synchronize()
    first = y8.clone()
    poison = [torch.full((c.dim * k * 5,), 7.0, device="cuda", dtype=torch.float32) for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(2):
        y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
    assert all(bool((p == 7.0).all()) for p in poison)
    c.apply_H(x8, y8, 8, N.BS_F32)
    torch.cuda.synchronize()
    assert torch.equal(y8, first)
    c.sync_status()
    del g
    c.close()
