"""The outer product A z of FGMRES on the two ways it takes (one kernel that converts the cycle's result while it
gathers, or a conversion and a product), at sizes around the line between them (10,240 entries per SM) and with short
and long rows: one Arnoldi step against the same step written out from the preconditioner's own result."""
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


P1 = dict(cf_mode=1, interp=1, lump_tol=0.05)
SYSTEMS = {
    "fd2d_40": lambda: W.fd_adr_2d(40, 0.6, 1e-3, 0.1), "fd2d_558": lambda: W.fd_adr_2d(558, 0.6, 1e-3, 0.1),
    "fd2d_559": lambda: W.fd_adr_2d(559, 0.6, 1e-3, 0.1), "fd3d_53": lambda: W.fd_adr_3d(53, (1.0, 0.7, 0.4), 1e-3, 0.1),
    "fd3d_66": lambda: W.fd_adr_3d(66, (1.0, 0.7, 0.4), 1e-3, 0.1), "dg_20": lambda: W.dg_p2_advection(20),
    "dg_110": lambda: W.dg_p2_advection(110),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_one_arnoldi_step(lair, name, precision):
    import torch
    s = SYSTEMS[name]()
    A = s.to_scipy()
    # 4^k entries of +-1: |b| is a power of two, so b / |b| is exact and the step's cycle is that of precond(b / |b|)
    k = int(np.log2(s.n) // 2)
    rng = np.random.default_rng(3)
    b = np.zeros(s.n)
    b[rng.permutation(s.n)[:4 ** k]] = rng.choice([-1.0, 1.0], 4 ** k)
    v = b / 2.0 ** k
    G = lair.Hierarchy.from_system(s, device=True, precision=precision, **P1)
    x, rep = G.solve(torch.from_numpy(b).cuda(), tol=0.0, cycle=lair.FGMRES, max_iter=1)
    assert rep.iters == 1
    z = G.precond(torch.from_numpy(v).cuda()).cpu().numpy()
    w = A @ z
    h0 = v @ w
    h1 = np.linalg.norm(w - h0 * v)
    want = 2.0 ** k * h0 / (h0 * h0 + h1 * h1) * z
    # z is the same to the bit; the rest are FP64 sums of up to n products with n 2^-53 < 2e-11, taken a few times
    assert np.abs(x.cpu().numpy() - want).max() <= 1e-10 * np.abs(want).max()
