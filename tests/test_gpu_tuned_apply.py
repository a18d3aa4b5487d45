"""Launch shapes that a caller sets, or the autotuner chooses, are the ones a
direct apply runs.  X-inverse forms 0, 1 and 2 agree bit for bit, and form 3 adds
in another order, which is how they are told apart."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu


def applied(plan, x, **shape):
    if shape:
        plan.set_tune(**shape)
    return plan.apply_preconditioner(x, precision=1)


@pytest.mark.parametrize("shape", [(16, 512), (40, 64), (256, 256)])
def test_x_inverse_form_zero_is_not_replaced(shape):
    import torch
    hz = hz_module()
    med, _ = media(hz, S.small_problem(shape, 4, M=5, Mt=3, width=3), oracle=False)
    plan = hz.Plan(med, precision=1, restart=1, max_nrhs=2)
    x = torch.from_numpy(S.random_field(np.random.default_rng(1), shape, 2)).cuda()
    zero, one, three = (applied(plan, x, rowinv_mode=m) for m in (0, 1, 3))
    assert torch.equal(zero, one)
    assert not torch.equal(zero, three)


def test_autotuned_apply_is_not_slower_than_the_default():
    """The default that the report states is what an untuned plan's apply
    takes, and the tuned plan keeps it where no candidate is faster."""
    hz = hz_module()
    med, _ = media(hz, S.small_problem((128, 128, 128), 4, M=6, Mt=2, width=6), oracle=False)
    plan = hz.Plan(med, precision=1, restart=2, max_nrhs=4)
    r = plan.autotune()
    assert 0 < r["apply_us"] <= r["apply_us_default"]
