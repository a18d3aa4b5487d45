"""Infinities in an Arnoldi step end the solve: with a right-hand side of norm
2e-155 (its square is still a number) the reciprocal of the residual's squared
norm, by which the projections are scaled, overflows.  The solve reports a
breakdown and leaves the initial guess as it is."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(precision=0), dict(precision=1), dict(precision=0, no_precond=True)])
@pytest.mark.parametrize("shape", [(16, 24), (64, 96)])
def test_overflowing_scale_is_a_breakdown(shape, opts):
    hz = hz_module()
    p = S.small_problem(shape, 11, M=3, Mt=2, width=2)
    med = hz.Medium(p.c, p.zeta, omega=p.omega, M=p.M, Mt=p.Mt, c_o=p.c_o)
    f = np.zeros((2,) + shape, complex)
    f[0, 5, 7] = 2e-155
    f[1] = S.random_field(np.random.default_rng(1), shape)
    plan = hz.Plan(med, restart=40, maxit=1000, max_nrhs=2, **opts)
    u, stats = plan.solve(f)
    assert stats[0]["status"] == 5 and not stats[0]["converged"]
    assert (u[0] == 0).all()
    if not opts.get("no_precond"):
        assert stats[1]["converged"]  # the other one goes on
