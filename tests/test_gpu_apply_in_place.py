"""Applies whose output is their input: bit for bit what they give elsewhere, in
both precisions, at sizes that take each form of the x-inverse (the one that adds
into an output cleared by the first pass among them) and of the symbol pass."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 512), (40, 64), (256, 256), (12, 8), (24, 2400), (512, 1024), (32, 24, 40),
                                   (128, 96, 96)])
@pytest.mark.parametrize("precision", [0, 1])
def test_in_place(shape, precision):
    import torch
    hz = hz_module()
    med, _ = media(hz, S.small_problem(shape, 4, M=5, Mt=3, width=3), oracle=False)
    plan = hz.Plan(med, precision=precision, restart=1, max_nrhs=2)
    x = torch.from_numpy(S.random_field(np.random.default_rng(3), shape, 2)).cuda()
    y = plan.apply_preconditioner(x, precision=precision)
    z = x.clone()
    plan.apply_preconditioner(z, precision=precision, out=z)
    assert torch.equal(y, z)
