"""Solves that replay the captured cycle at the benchmark workloads' full sizes.
A plan runs its first three full cycles step by step, so the solve is repeated
until its cycles come from the graph (seen in the phase profile, which a replay
leaves empty); the solution is then bit for bit that of the direct launches, and
meets the tolerance by the oracle's operator."""
import numpy as np
import pytest

import oracle as O
from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,alpha,checked", [("config2", 0.1, (0,)), ("config4", 0.1, (0, 31, 63))])
def test_replayed_solve(name, alpha, checked):
    import torch
    hz = hz_module()
    p = getattr(S, name)()
    med, med_o = media(hz, p, alpha=alpha)
    plan = hz.Plan(med, precision=1, restart=p.restart, tol=p.tol, max_nrhs=p.f.shape[0], graphs=True)
    plan.autotune()
    f = torch.from_numpy(np.ascontiguousarray(p.f)).cuda()
    first, st = plan.solve(f)
    plan.solve(f)
    hz.profile_enable(True)
    hz.profile_read(reset=True)
    try:
        u, st_replay = plan.solve(f)
        phases = hz.profile_read(reset=True)
    finally:
        hz.profile_enable(False)
    for phase in ("cgs2_dots", "givens"):
        assert phases.get(phase, {"launches": 0})["launches"] == 0, phases
    assert torch.equal(u, first)
    assert [s["iters"] for s in st] == [s["iters"] for s in st_replay]
    u = u.cpu().numpy()
    for b in checked:
        r = rel(O.apply_operator(med_o, u[b]), p.f[b])
        assert st_replay[b]["converged"] and r <= p.tol, (b, r)
