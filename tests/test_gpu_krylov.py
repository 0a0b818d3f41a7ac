"""The outer FGMRES reductions at the ends of their variants: restart lengths around 8, 16 and 24 columns and the
longest, sizes around a block's elements, one system and a batch."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lair():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1708_06065_gb300 import lair as L
    torch.cuda.init()
    return L


OPTS = dict(cf_mode=1, interp=1, lump_tol=0.05)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("restart", [1, 8, 9, 16, 17, 24, 25, 31])
@pytest.mark.parametrize("N", [16, 23, 60])
def test_restart_lengths(lair, N, restart, precision):
    import torch
    # diffusion with one-point interpolation: slow enough for a full restart cycle
    s = W.fd_adr_2d(N, 0.7, 0.5, 0.1, b_seed=N)
    A = s.to_scipy()
    kw = dict(OPTS, precision=precision, fgmres_restart=restart, coarse_max=8)
    b = torch.from_numpy(s.b).cuda()
    # the residual that stops the iteration is b - A x in FP64: recomputed here it differs by rounding only
    lim = 1e-9 * (1 + 1e-6)
    G = lair.Hierarchy.from_system(s, device=True, **kw)
    x, rep = G.solve(b, tol=1e-9, cycle=lair.FGMRES, max_iter=2000)
    assert rep.status == 0 and np.linalg.norm(s.b - A @ x.cpu().numpy()) <= lim * np.linalg.norm(s.b)
    two, offs = W.block_diagonal([s, W.fd_adr_2d(N + 1, 0.2, 1e-3, 0.1, b_seed=1)])
    dev = [torch.from_numpy(a).cuda() for a in (two.row_ptr, two.col, two.val, two.b)]
    B = lair.Hierarchy.batched(*dev[:3], offs, **kw)
    xb, its, rel, st = B.solve_batched(dev[3], tol=1e-9, cycle=lair.FGMRES, max_iter=2000)
    assert st == 0 and rel.max() <= 1e-9
    r = two.b - two.to_scipy() @ xb.cpu().numpy()
    for q in range(2):
        sl = slice(offs[q], offs[q + 1])
        assert np.linalg.norm(r[sl]) <= lim * np.linalg.norm(two.b[sl])
