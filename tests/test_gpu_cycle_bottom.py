"""The V-cycle's kernels for levels that fit on the GPU at once. The smallest levels run in one CTA (matrix entries and
vectors in shared memory, the coarsest product over a cluster), the others with one row per thread: sizes around the
limits (1,024 rows in the first bottom level, 512 unknowns in the coarsest, entries that do not fit in shared memory,
rows longer than the entries read ahead), every sweep order; after a refresh, and for a batch."""
import numpy as np
import pytest

import workloads as W
from helpers import entrywise_rel, with_values
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


P1 = dict(cf_mode=1, interp=1, lump_tol=0.05)
CASES = [
    (24, dict(coarse_max=1)), (24, dict(P1, coarse_max=300)), (33, dict(coarse_max=512)), (45, dict(coarse_max=513)),
    (45, dict(P1)), (46, dict(P1)), (58, dict()), (90, dict()), (130, dict()), (150, dict(P1, coarse_max=8)),
    (60, dict(P1, coarse_max=700)), (60, dict(P1, relax=2, coarse_max=700)),   # no bottom: split results down to the coarsest
    (181, dict(distance=2, lump_tol=0.0)), (64, dict(cf_mode=0, relax=1)), (64, dict(cf_mode=0, relax=2)),
    (100, dict(P1, relax=1)), (100, dict(P1, relax=2)),
]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,kw", CASES)
def test_cycle_with_small_levels_matches_oracle(lair, N, kw, precision):
    import torch
    s = W.fd_adr_2d(N, 0.6, 1e-3, 0.1, b_seed=3)
    G = lair.Hierarchy.from_system(s, device=True, precision=precision, **kw)
    H = O.Hierarchy(s, prec=precision, **kw)
    assert [i["n"] for i in G.info()] == [L.n for L in H.levels]
    # every row is summed in the oracle's order; only the coarsest level differs (inverse against LU solve)
    tol = 1e-10 if precision == 0 else 1e-5
    for seed in (0, 1):
        v = np.random.default_rng(seed).uniform(-1, 1, s.n)
        z = G.precond(torch.from_numpy(v).cuda()).cpu().numpy()
        assert entrywise_rel(z, H.precond(v)) <= tol
    # the packed images follow a refresh
    val = s.val * np.random.default_rng(5).uniform(0.9, 1.1, s.nnz)
    G.refresh(val)
    H.refresh(with_values(s, val))
    assert entrywise_rel(G.precond(torch.from_numpy(v).cuda()).cpu().numpy(), H.precond(v)) <= tol


@pytest.mark.parametrize("sides", [(20,), (33, 64, 17), (90, 90, 45)])
def test_batched_cycle_with_small_levels(lair, sides):
    import torch
    systems = [W.fd_adr_2d(n, 0.3 + k, 1e-2, 0.2, b_seed=k) for k, n in enumerate(sides)]
    s, offs = W.block_diagonal(systems)
    dev = [torch.from_numpy(a).cuda() for a in (s.row_ptr, s.col, s.val, s.b)]
    G = lair.Hierarchy.batched(*dev[:3], offs, **P1)
    x, _, rel, st = G.solve_batched(dev[3], cycle=lair.FGMRES, tol=1e-10)
    assert st == 0 and rel.max() <= 1e-10
    import scipy.sparse.linalg as sl
    assert entrywise_rel(x.cpu().numpy(), sl.spsolve(s.to_scipy().tocsc(), s.b)) <= 1e-6


def test_precond_on_overlapping_vectors(lair):
    """x = M^-1 b written over b, and over a vector that shares half of it: the same as into a vector of its own."""
    import torch
    s = W.fd_adr_2d(70, 0.6, 1e-3, 0.1)
    for precision in (0, 1):
        G = lair.Hierarchy.from_system(s, device=True, precision=precision, **P1)
        v = torch.from_numpy(np.random.default_rng(2).uniform(-1, 1, s.n)).cuda()
        z = G.precond(v)
        own = v.clone()
        assert torch.equal(G.precond(own, own), z)
        buf = torch.zeros(s.n + s.n // 2, dtype=torch.float64, device="cuda")
        buf[:s.n] = v
        assert torch.equal(G.precond(buf[:s.n], buf[s.n // 2:]), z)
