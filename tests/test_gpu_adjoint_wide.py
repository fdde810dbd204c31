"""Adjoint in wide spaces: 34 states per species, past the Gram tables (densities by jumps), and sd + pf (32 states), whose
pair matrices take several 64 x 64 tiles.  Every seventh to fortieth parameter against the oracle's unit-parameter matrices;
tolerances as derived in test_gpu_adjoint_edges.py: (k + 1) 2^-24 sum |gy| |H_t| |x| for FP32, 10^6 2^-53 for FP64."""
import numpy as np
import pytest

import oracle as O
from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

J34 = [I.Orbit(0, 8, 17), I.Orbit(0, 8, 15)]
SDPF = list(I.SD_ORBITS) + list(I.PF_ORBITS)


_unit = {}


def unit(orbits, Z, Nn, twoM, spe, tb, t):
    key = (len(orbits), Z, Nn, t)
    if key not in _unit:
        e = np.zeros(len(spe))
        e[t:t + 1] = 1.0
        o = O.Oracle(orbits, Z, Nn, twoM, 0)
        _unit[key] = o.set_interaction(e, [(*tb[t - len(spe)][:6], 1.0)] if t >= len(spe) else []).matrix()
    return _unit[key]


@pytest.mark.parametrize("orbits,Z,Nn,twoM,step", [(J34, 1, 1, 0, 7), (J34, 2, 1, 1, 10), (J34, 1, 2, 3, 10), (SDPF, 1, 1, 0, 40),
                                                   (SDPF, 2, 1, 1, 40), (SDPF, 1, 2, 1, 40)])
@pytest.mark.parametrize("k,dtype", [(1, N.BS_F32), (4, N.BS_F32), (8, N.BS_F32), (1, N.BS_F64), (8, N.BS_F64)])
def test_some_parameters(orbits, Z, Nn, twoM, step, k, dtype):
    spe, tb = [0.5 * i - 1.0 for i in range(len(orbits))], I.random_tbmes(orbits)
    c = N.make(orbits, spe, tb, Z, Nn, twoM, +1, device=0)
    tdt = torch.float64 if dtype == N.BS_F64 else torch.float32
    x, gy = (torch.from_numpy(I.random_block(c.dim, k, seed=s)).to("cuda", tdt) for s in (3, 4))
    n = len(spe) + len(tb)
    g = c.apply_H_backward(x, gy, torch.empty_like(gy), k, dtype, n_theta=n)
    c.close()
    xh, gh = x.double().cpu().numpy(), gy.double().cpu().numpy()
    rel = (k + 1) * 2.0 ** -24 if dtype == N.BS_F32 else 1e6 * 2.0 ** -53
    for t in range(0, n, step):
        H = unit(orbits, Z, Nn, twoM, spe, tb, t)
        tol = rel * np.sum(np.abs(gh) * (abs(H) @ np.abs(xh))) + 1e-300
        assert abs(g[t] - np.sum(gh * (H @ xh))) <= tol, t


@pytest.mark.parametrize("orbits,Z,Nn,twoM,step", [(J34, 2, 1, 1, 10), (J34, 1, 2, 3, 10), (list(I.SD_ORBITS), 2, 2, 0, 5)])
@pytest.mark.parametrize("keep", [0, 3])
@pytest.mark.parametrize("k,dtype", [(4, N.BS_F32), (1, N.BS_F64)])
def test_elements_of_value_zero(orbits, Z, Nn, twoM, step, keep, k, dtype):
    """Gradients do not depend on the elements' values: all zero, or all but every third."""
    spe = [0.5 * i - 1.0 for i in range(len(orbits))]
    tb = [(*t[:6], t[6] if keep and n % keep == 0 else 0.0) for n, t in enumerate(I.random_tbmes(orbits))]
    c = N.make(orbits, spe, tb, Z, Nn, twoM, +1, device=0)
    tdt = torch.float64 if dtype == N.BS_F64 else torch.float32
    x, gy = (torch.from_numpy(I.random_block(c.dim, k, seed=s)).to("cuda", tdt) for s in (3, 4))
    n = len(spe) + len(tb)
    g = c.apply_H_backward(x, gy, torch.empty_like(gy), k, dtype, n_theta=n)
    c.close()
    xh, gh = x.double().cpu().numpy(), gy.double().cpu().numpy()
    rel = (k + 1) * 2.0 ** -24 if dtype == N.BS_F32 else 1e6 * 2.0 ** -53
    for t in range(0, n, step):
        H = unit(orbits, Z, Nn, twoM, spe, tb, t)
        tol = rel * np.sum(np.abs(gh) * (abs(H) @ np.abs(xh))) + 1e-300
        assert abs(g[t] - np.sum(gh * (H @ xh))) <= tol, t
