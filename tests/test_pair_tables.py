"""Host tables of the pair-core pn kernel (bs_pair.cpp), checked on the CPU:
walking them as the kernel does, with the like-particle terms from the
destination lists, gives the same H x as the general tables (which
test_host_tables.py pins to the oracle), and every index stays inside its
buffer."""
import numpy as np
import pytest

from paper_1801_08432_gb300 import _native as N
from paper_1801_08432_gb300 import inputs as I
from tests.test_host_tables import tables_matvec

REC = np.dtype([("xoff", np.uint32), ("yoff", np.uint32), ("srec", np.uint32), ("wj", np.uint32)])
ROW = np.dtype([("elem", np.int64), ("ycol", np.int32), ("n", np.int32), ("part", np.int32), ("state", np.int32),
                ("sign", np.int32), ("pad", np.int32)])
TILE = np.dtype([("rec0", np.int32), ("nrec", np.int32), ("core0", np.int32), ("ncore", np.int32), ("woff", np.int32),
                 ("np", np.int32), ("row0", np.uint16, 4), ("nrow", np.uint8, 4),
                 ("first", np.uint16, 4), ("pad", np.int32)])
ITEM = np.dtype([(n, np.int32) for n in ("rec0", "nrec", "tile0", "ntile", "row0", "nrow", "store0", "nstore", "cols")]
                + [("pad", np.int32, 3)])


def tables(c, cp):
    get = lambda name, dt: np.frombuffer(c.table(name, np.uint8).tobytes(), dtype=dt)
    return (get("pr_items%d" % cp, ITEM), get("pr_tiles%d" % cp, TILE), get("pr_rows%d" % cp, REC),
            get("pr_store%d" % cp, ROW))


def pair_matvec(c, x, Z, cp):
    """The pn term of y = H x from the pair tables, with the kernel's tiles, groups and rounds."""
    nsign = c.table("pr_nsign", np.uint32)
    colpos = c.table("pr_colpos", np.uint16).reshape(-1, len(nsign))
    w = c.table("pr_w", np.float64)
    recs = np.frombuffer(c.table("pr_recs", np.uint8).tobytes(), dtype=REC)
    items, tiles, rows, store = tables(c, cp)
    part = np.zeros((Z, len(x)))
    written = np.zeros((Z, len(x)), dtype=int)
    for it in items:
        R = recs[it["rec0"]:it["rec0"] + it["nrec"]]
        J = rows[it["row0"]:it["row0"] + it["nrow"]]
        Y = np.zeros(it["cols"])
        owner = np.full(it["cols"], -1)
        for t in tiles[it["tile0"]:it["tile0"] + it["ntile"]]:
            assert 0 < t["ncore"] <= 128 and t["core0"] + t["ncore"] <= len(nsign)
            assert t["rec0"] + t["nrec"] <= it["nrec"] and np.all(t["nrow"] <= 16)
            cores = np.arange(t["core0"], t["core0"] + t["ncore"])
            K = R[t["rec0"]:t["rec0"] + t["nrec"]]
            W = w[t["woff"]:t["woff"] + t["np"] ** 2].reshape(t["np"], t["np"])
            X = np.zeros((len(K), len(cores)))
            for a, r in enumerate(K):
                l = int(r["wj"] >> 16 & 255)
                assert int(r["srec"] & 31) == 31 - l
                col = colpos[l, cores]
                ok = col != 0xFFFF
                s = np.where((nsign[cores] >> np.uint32(l)) & 1, -1.0, 1.0) * (-1.0 if r["srec"] >> 31 else 1.0)
                X[a, ok] = (s * x[np.where(ok, r["xoff"] + col.astype(np.int64), 0)])[ok]
            for g in range(4):   # consumer groups
                hit, last, first = set(), 0, int(t["nrow"][g] > 0)
                for n, r in enumerate(J[t["row0"][g]:t["row0"][g] + t["nrow"][g]]):
                    l, rd = int(r["wj"] >> 16 & 255), int(r["wj"] >> 24)
                    assert rd >= last and int(r["srec"] & 31) == 31 - l   # in the order of their rounds
                    first |= (n > 0 and rd > last) << n
                    last = rd
                    col = colpos[l, cores]
                    ok = col != 0xFFFF
                    at = int(r["yoff"]) + col[ok].astype(int)
                    assert at.size == 0 or at.max() < it["cols"]
                    assert np.all((owner[at] == -1) | (owner[at] == g))   # one group per element
                    owner[at] = g
                    assert not hit & {(rd, q) for q in at.tolist()}       # one add per element and round
                    hit |= {(rd, q) for q in at.tolist()}
                    s = np.where((nsign[cores] >> np.uint32(l)) & 1, -1.0, 1.0)
                    Y[at] += (s * (W[(K["wj"] & 0xFFFF).astype(int), int(r["wj"] & 0xFFFF)] @ X))[ok]
                assert first == t["first"][g]
        for r in store[it["store0"]:it["store0"] + it["nstore"]]:
            y = Y[r["ycol"]:r["ycol"] + r["n"]]
            assert len(y) == r["n"] and 0 <= r["part"] < Z
            part[r["part"], r["elem"]:r["elem"] + r["n"]] = -y if r["sign"] else y
            written[r["part"], r["elem"]:r["elem"] + r["n"]] += 1
    assert np.all(written == 1)   # every element of every partial vector, once
    return part.sum(axis=0)


SPACES = [("sd", 2, 2, 0), ("sd", 3, 2, 1), ("sd", 1, 1, 0), ("sd", 5, 1, 2), ("p", 3, 3, 0),
          ("pf", 2, 2, 2), ("pf", 2, 1, 1)]


@pytest.mark.parametrize("name,Z,Nn,twoM", SPACES)
@pytest.mark.parametrize("cp", [1, 4])
def test_pair_tables_reproduce_the_pn_term(name, Z, Nn, twoM, cp):
    orbits, spe, tb = I.space(name)
    par = (-1) ** (((Z + Nn) * (orbits[0].l % 2)) % 2)
    c = N.make(orbits, spe, tb, Z, Nn, twoM, par, device=-1)
    x = I.random_block(c.dim, 1, seed=5)[:, 0]
    y = pair_matvec(c, x, Z, cp) + like_matvec(c, x)
    ref = tables_matvec(c, x)
    assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))


def like_matvec(c, x):
    """The pp and nn terms of y = H x from the destination lists."""
    B = c.export_basis()
    pp, pps, ppc = c.table("pp_ptr", np.int64), c.table("pp_src", np.int32), c.table("pp_coef", np.float64)
    nn, nns, nnc = c.table("nn_ptr", np.int64), c.table("nn_src", np.int32), c.table("nn_coef", np.float64)
    y = np.zeros_like(x)
    V = lambda a, b: a[int(B["blocks"][b][2]):][:shape(b)[0] * shape(b)[1]].reshape(shape(b))
    shape = lambda b: (int(B["p_sec"][B["blocks"][b][0]][3]), int(B["n_sec"][B["blocks"][b][1]][3]))
    for b, (ps, ns_, off) in enumerate(B["blocks"]):
        X, Y = V(x, b), V(y, b)
        p0, n0 = int(B["p_sec"][ps][2]), int(B["n_sec"][ns_][2])
        for r in range(X.shape[0]):
            e = slice(pp[p0 + r], pp[p0 + r + 1])
            Y[r] += ppc[e] @ X[pps[e]]
        for q in range(X.shape[1]):
            e = slice(nn[n0 + q], nn[n0 + q + 1])
            Y[:, q] += X[:, nns[e]] @ nnc[e]
    return y
