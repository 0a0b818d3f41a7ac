"""Launch schedules of the cycle's large views. A view is tuned when its launch in the cycle, copied rows included, is
above what the kernels with one schedule take (2,048 rows per SM in FP32, 1,024 in FP64), and the choice never changes
a result."""
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
# 96^3 mixed: sweeps that copy nothing (F) and that carry the F rows along (C). 512^2 with lAIP in FP64: about 131,000 F
# rows, which alone would be below the limit of 152 SMs, and as many copied ones; P has all rows.
CASES = [("fd3d", 96, dict(P1, precision=1), {"sweep_F", "sweep_C"}),
         ("fd3d", 80, dict(P1, precision=0), {"sweep_F", "sweep_C"}),
         ("fd2d", 512, dict(precision=0), {"sweep_F", "sweep_C", "interp"})]


@pytest.mark.parametrize("family,N,kw,kernels", CASES)
def test_large_views_are_tuned_and_keep_every_bit(lair, family, N, kw, kernels):
    import torch
    s = W.fd_adr_3d(N, (1.0, 0.7, 0.4), 1e-5, 0.05) if family == "fd3d" else W.fd_adr_2d(N, 0.6, 1e-4, 0.1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    G0 = lair.Hierarchy.from_system(s, device=True, autotune=0, timing=1, **kw)
    G1 = lair.Hierarchy.from_system(s, device=True, autotune=1, timing=1, **kw)
    assert not [k for k in G0.timers() if k.startswith("tune_L")]
    tuned = {k.split(":")[0] for k in G1.timers() if k.startswith("tune_L")}
    # expected from the level sizes alone
    limit = sms * (2048 if kw["precision"] == 1 else 1024)
    want, p1 = set(), kw.get("interp") == 1
    for l, i in enumerate(G1.info()[:-1]):
        F, C = i["n"] - i["nc"], i["nc"]
        launches = {"restrict": (C, 0), "sweep_F": (F, 0 if p1 else C), "sweep_C": (C, 0 if p1 and l else F)}
        if not p1:
            launches["interp"] = (F + C, 0)
        want |= {f"tune_L{l}_{k}" for k, (rows, copied) in launches.items() if rows >= 65536 and rows + copied > limit}
    assert tuned == want and {f"tune_L0_{k}" for k in kernels} <= tuned
    v = torch.from_numpy(np.random.default_rng(2).uniform(-1, 1, s.n)).cuda()
    assert torch.equal(G0.precond(v), G1.precond(v))
    b = torch.from_numpy(s.b).cuda()
    x0, r0 = G0.solve(b, tol=1e-8)
    x1, r1 = G1.solve(b, tol=1e-8)
    assert r0.status == 0 and r0.iters == r1.iters and torch.equal(x0, x1)
    # a second hierarchy takes the choices without timing
    G2 = lair.Hierarchy.from_system(s, device=True, timing=1, **kw)
    again = {k for k in G2.timers() if k.startswith("tune_L")}
    assert {k.split(":")[0] for k in again} == want and all(k.endswith(" cached") for k in again)
