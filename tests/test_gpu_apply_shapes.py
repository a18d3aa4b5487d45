"""Untuned complex64 applies take their shape by size: every shape of the rule
against the oracle, with tiles that end inside the grid, on plans whose
right-hand-side count reaches the rule's sizes (the call itself has two)."""
import numpy as np
import pytest

import oracle as O
from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media, rel, within

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,max_nrhs,basis", [
    ((256, 24), 700, 0), ((128, 60), 600, 0), ((256, 12, 20), 80, 0), ((256, 40), 500, 2),  # node loop
    ((512, 16), 300, 0), ((64, 48), 700, 0),                    # four nodes per block
    ((96, 20), 2, 0), ((96, 48), 100, 0),                       # one column, half blocks
    ((120, 24), 2, 0), ((180, 32), 800, 0),                     # factor 5: one column, four nodes
    ((16, 512), 2, 0), ((40, 64), 2, 0)])                       # x-inverse line by line
def test_against_the_oracle(shape, max_nrhs, basis):
    import torch
    hz = hz_module()
    p = S.small_problem(shape, 4, M=5, Mt=3, width=3)
    med, med_o = media(hz, p, basis=basis)
    rng = np.random.default_rng(8)
    v = np.stack([S.random_field(rng, shape) for _ in range(2)])
    plan = hz.Plan(med, precision=1, restart=1, max_nrhs=max_nrhs)
    y = plan.apply_preconditioner(torch.from_numpy(v).cuda(), precision=1).cpu().numpy()
    for b in range(2):
        assert within(rel(y[b], O.apply_preconditioner(med_o, v[b])), 1, "interp_small")
