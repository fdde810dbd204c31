"""Pair tables with neutron groups of more than 128 cores (three pf neutrons: up to 145): a group's cores in two tiles."""
import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I
from tests.test_host_tables import tables_matvec
from tests.test_pair_tables import like_matvec, pair_matvec, tables


@pytest.mark.parametrize("Z,Nn,twoM", [(1, 4, 1), (2, 4, 0)])
@pytest.mark.parametrize("cp", [1, 4])
def test_groups_of_two_tiles(Z, Nn, twoM, cp):
    orbits, spe, tb = I.space("pf")
    c = N.make(orbits, spe, tb, Z, Nn, twoM, (-1) ** ((Z + Nn) % 2), device=-1)
    tiles_ = tables(c, cp)[1]
    assert any(a["core0"] + a["ncore"] == b["core0"] and a["rec0"] == b["rec0"] and np.array_equal(a["row0"], b["row0"])
               for a, b in zip(tiles_[:-1], tiles_[1:]))   # a second tile of the same rows
    x = I.random_block(c.dim, 1, seed=5)[:, 0]
    y = pair_matvec(c, x, Z, cp) + like_matvec(c, x)
    ref = tables_matvec(c, x)
    assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))
