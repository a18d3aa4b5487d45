"""A plan for very many right-hand sides of a small grid keeps the symbol pass's
plain form, which suits a call with few of them too.  The looped form's results
differ in their last bits, which is how the two are told apart."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,max_nrhs", [((256, 256), 64), ((128, 128), 256), ((64, 64), 1024)])
def test_many_small_grids_keep_the_plain_symbol_pass(shape, max_nrhs):
    """More than 2^22 points over a plan's right-hand sides, but too few in one
    for blocks that loop over nodes."""
    import torch
    hz = hz_module()
    med, _ = media(hz, S.small_problem(shape, 4, M=5, Mt=3, width=3), oracle=False)
    plan = hz.Plan(med, precision=1, restart=1, max_nrhs=max_nrhs)
    x = torch.from_numpy(S.random_field(np.random.default_rng(1), shape, 2)).cuda()
    untuned = plan.apply_preconditioner(x, precision=1)
    plan.set_tune(syminv_kpb=1, col_pair=1, rowinv_mode=0)
    assert torch.equal(untuned, plan.apply_preconditioner(x, precision=1))
