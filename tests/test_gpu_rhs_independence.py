"""A right-hand side's apply does not depend on how many are in the call, bit
for bit, in both precisions: grids on both sides of the size at which blocks of
one line (or a quarter of the columns) fill the GPU better, counts at which the
call as a whole would be on the other side."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(96, 128), (128, 128), (240, 360), (48, 40, 24), (64, 64, 64), (20, 512)])
@pytest.mark.parametrize("precision", [0, 1])
def test_alone_and_in_company(shape, precision):
    import torch
    hz = hz_module()
    p = S.small_problem(shape, 4, M=5, Mt=3, width=3)
    med, _ = media(hz, p, oracle=False)
    plan = hz.Plan(med, precision=precision, restart=1, max_nrhs=8)
    x = torch.from_numpy(S.random_field(np.random.default_rng(2), shape, 8)).cuda()
    whole = plan.apply_preconditioner(x, precision=precision)
    for k in (1, 2, 3):
        part = plan.apply_preconditioner(x[:k].contiguous(), precision=precision)
        assert torch.equal(part, whole[:k]), k
    assert torch.equal(plan.apply_preconditioner(x[5:6].contiguous(), precision=precision), whole[5:6])
