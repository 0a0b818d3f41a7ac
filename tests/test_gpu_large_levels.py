"""One-point hierarchies whose finest levels are above the one-wave kernels' limits (152 SMs: 155,648 rows in FP64,
311,296 in FP32): interpolation into both x buffers and sweeps that copy nothing, tuned, against the oracle's cycle,
before and after a refresh."""
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


@pytest.mark.parametrize("N,precision,relax", [(71, 0, 0), (90, 1, 0), (71, 0, 2)])
def test_cycle_and_refresh_match_oracle(lair, N, precision, relax):
    import torch
    s = W.fd_adr_3d(N, (1.0, 0.7, 0.4), 1e-5, 0.05)
    kw = dict(cf_mode=1, interp=1, lump_tol=0.05, precision=precision, relax=relax)
    G = lair.Hierarchy.from_system(s, device=True, **kw)
    kw.pop("precision")
    H = O.Hierarchy(s, prec=precision, **kw)
    n, nc = G.info()[0]["n"], G.info()[0]["nc"]
    assert [i["n"] for i in G.info()] == [L.n for L in H.levels]
    # both sweeps' views of the finest level are above the limit, or their rows and copies are
    assert n - nc > 152 * (2048 if precision else 1024) and n > n - nc
    # every row is summed in the oracle's order; only the coarsest level differs (inverse against LU solve)
    tol = 1e-10 if precision == 0 else 1e-5
    v = np.random.default_rng(1).uniform(-1, 1, s.n)
    dv = torch.from_numpy(v).cuda()
    assert entrywise_rel(G.precond(dv).cpu().numpy(), H.precond(v)) <= tol
    val = s.val * np.random.default_rng(5).uniform(0.95, 1.05, s.nnz)
    G.refresh(val)
    H.refresh(with_values(s, val))
    assert entrywise_rel(G.precond(dv).cpu().numpy(), H.precond(v)) <= tol
    b = torch.from_numpy(s.b).cuda()
    x, rep = G.solve(b, tol=1e-8)
    r = s.b - with_values(s, val).to_scipy() @ x.cpu().numpy()
    assert rep.status == 0 and np.linalg.norm(r) <= 1e-8 * (1 + 1e-6) * np.linalg.norm(s.b)
