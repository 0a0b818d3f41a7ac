"""The algorithmic bytes of the one-point interpolation: a column and a result per row, a coarse value per entry, and a
second write of the C points on levels whose sweeps copy nothing (F-F-C; the other orders copy)."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("relax,second", [(0, True), (1, False), (2, False)])
def test_interpolation_bytes(precision, relax, second):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1708_06065_gb300 import lair
    s = W.fd_adr_2d(120, 0.6, 1e-3, 0.1)
    G = lair.Hierarchy.from_system(s, device=True, cf_mode=1, interp=1, lump_tol=0.05, precision=precision, relax=relax,
                                   timing=1)
    G.solve(torch.from_numpy(s.b).cuda(), tol=1e-6)
    i, sv = G.info()[0], 4 if precision else 8
    want = i["n"] * (4 + sv) + (i["nnz_P"] + (i["nc"] if second else 0)) * sv
    assert G.timers()["L0_interp"][2] == want
