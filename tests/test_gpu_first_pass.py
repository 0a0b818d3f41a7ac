"""The first pass against the oracle where one of its paths ends: rows of ST with 31, 32 and more than 127
dependants, rows of S longer than the eight lanes that share one, several blocks (staged graphs, and more blocks than
SMs, read through the cache), points without any strong connection."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lair():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1708_06065_gb300 import lair as L
    torch.cuda.init()
    return L


def star(hubs, leaves):
    """hubs points with `leaves` dependants each, the leaves in a chain, and isolated points between them."""
    n = hubs * (leaves + 2)
    rows, cols, vals = [], [], []
    for h in range(hubs):
        o = h * (leaves + 2)
        for k in range(leaves):
            rows += [o + 1 + k, o + 1 + k]
            cols += [o, o + 1 + (k + 1) % leaves]
            vals += [-1.0, -0.9 - 0.001 * k]
        rows.append(o)
        cols.append((o + leaves + 2) % n)
        vals.append(-0.5)
    acc = {}
    for r, c, v in zip(rows, cols, vals):
        if r != c:
            acc[(r, c)] = acc.get((r, c), 0.0) + v
    rows, cols = (np.array(a) for a in zip(*acc))
    vals = np.array(list(acc.values()))
    r = np.concatenate([rows, np.arange(n)])
    c = np.concatenate([cols, np.arange(n)])
    v = np.concatenate([vals, np.full(n, 4.0)])
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return W.CsrSystem(n, rp.astype(np.int64), c[o].astype(np.int32), v[o], np.ones(n))


SYSTEMS = {
    "star30": lambda: star(9, 30), "star31": lambda: star(9, 31), "star32": lambda: star(7, 32),
    "star33": lambda: star(7, 33), "star100": lambda: star(5, 100),
    "star126": lambda: star(3, 126), "star127": lambda: star(3, 127), "star140": lambda: star(3, 140),
    "random": lambda: W.random_sparse(3000, 12, 4, sym_pattern=True), "wide": lambda: W.random_sparse(700, 40, 5),
    "fd2d": lambda: W.fd_adr_2d(90, 0.4, 1e-2, 0.1), "fd3d": lambda: W.fd_adr_3d(22, (1.0, 0.7, 0.4), 1e-3, 0.1),
    "chain": lambda: W.upwind_chain(257),
}


@pytest.mark.parametrize("rs_block", [64, 4096])
@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_first_pass_matches_oracle(lair, name, rs_block):
    s = SYSTEMS[name]()
    kw = dict(cf_mode=3, rs_block=rs_block, strength_abs=1, interp=1)
    G = lair.Hierarchy.from_system(s, device=True, **kw)
    H = O.Hierarchy(s, **kw)
    assert [i["n"] for i in G.info()] == [L.n for L in H.levels]
    for l in range(len(H.levels) - 1):
        assert np.array_equal(G.export_cf(l)[0], H.levels[l].cf), l


@pytest.mark.parametrize("n", [1022, 1023, 1024, 4095, 4096, 16382, 16383, 16384, 70000])
def test_scan_lengths(lair, n):
    """Level sizes at which the exclusive scans change from one kernel to the next."""
    s = W.upwind_chain(n)
    kw = dict(cf_mode=1, interp=1, strength_abs=1)
    G = lair.Hierarchy.from_system(s, device=True, **kw)
    H = O.Hierarchy(s, **kw)
    assert [i["n"] for i in G.info()] == [L.n for L in H.levels]
    for l in range(len(H.levels) - 1):
        assert np.array_equal(G.export_csr(l, 1)[0], H.levels[l].R[0]), l
        assert np.array_equal(G.export_csr(l + 1, 0)[0], H.levels[l + 1].A[0]), l
