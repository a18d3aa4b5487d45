"""The unpreconditioned method keeps small values: the solution after m steps
from a point source, whose field falls by many orders of magnitude from point to
point, against the same steps in extended precision, element by element."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module

L, CL = np.longdouble, np.clongdouble
# Each element has to be within TOL of the sum of the magnitudes of the terms
# y_j V_j that make it up.  FP64 Arnoldi (NumPy, below) is within 2e-14 of it.
TOL = 1e-11
CASES = [((64, 64), 24), ((60, 96), 30), ((16, 20, 24), 20)]


def problem(shape):
    p = S.small_problem(shape, 9, M=3, Mt=2, width=4)
    f = np.zeros((2,) + shape, complex)
    f[(0,) + tuple(n // 2 for n in shape)] = 1.0
    f[(1,) + tuple(n // 3 for n in shape)] = 0.5 - 2.0j
    return p, f


def gmres(p, f, m, real, cplx):
    """(u, sum of |y_j V_j|) after m steps of unpreconditioned GMRES (CGS2)."""
    c2, z, h2 = p.c * p.c, p.zeta, float(p.shape[-1]) ** 2
    g = (c2 * (1 - z * z) * h2).astype(real) + 1j * (-2 * c2 * z * h2).astype(real)
    rho = [real(float(n) ** 2 / h2) for n in p.shape]

    def apply_op(x):
        s = sum(rho[a] * (np.roll(x, 1, a) - 2 * x + np.roll(x, -1, a)) for a in range(x.ndim))
        return g * s + real(p.omega * p.omega) * x

    V = np.zeros((m + 1, f.size), cplx)
    R = np.zeros((m + 1, m), cplx)
    b = np.zeros(m + 1, cplx)
    b[0] = np.sqrt((abs(f) ** 2).sum())
    V[0] = f.ravel() / b[0]
    for j in range(m):
        w = apply_op(V[j].reshape(f.shape)).ravel()
        for _ in range(2):
            h = (V[:j + 1].conj() * w).sum(1)
            w = w - (h[:, None] * V[:j + 1]).sum(0)
            R[:j + 1, j] += h
        R[j + 1, j] = np.sqrt((abs(w) ** 2).sum())
        V[j + 1] = w / R[j + 1, j]
    for j in range(m):  # Givens rotations
        a, c = R[j, j], R[j + 1, j]
        r = np.sqrt(abs(a) ** 2 + abs(c) ** 2)
        G = np.array([[a.conj() / r, c.conj() / r], [-c / r, a / r]], cplx)
        R[j:j + 2] = G[:, :1] * R[j] + G[:, 1:] * R[j + 1]
        b[j:j + 2] = G[:, 0] * b[j] + G[:, 1] * b[j + 1]
    y = np.zeros(m, cplx)
    for i in range(m - 1, -1, -1):
        y[i] = (b[i] - (R[i, i + 1:m] * y[i + 1:]).sum()) / R[i, i]
    terms = V[:m] * y[:, None]
    return terms.sum(0).reshape(f.shape), abs(terms).sum(0).reshape(f.shape)


def test_fp64_arnoldi_is_well_within_the_tolerance():
    for shape, m in CASES:
        p, f = problem(shape)
        ref, size = gmres(p, f[0].astype(CL), m, L, CL)
        u, _ = gmres(p, f[0], m, np.float64, np.complex128)
        s = size > 0
        assert (abs(u - ref)[s] / size[s]).max() <= 0.1 * TOL
        assert size[s].min() <= 1e-8 * size.max()  # the case has small values


@pytest.mark.gpu
@pytest.mark.parametrize("shape,m", CASES)
def test_every_element(shape, m):
    hz = hz_module()
    p, f = problem(shape)
    med = hz.Medium(p.c, p.zeta, omega=p.omega, M=p.M, Mt=p.Mt, c_o=p.c_o)
    plan = hz.Plan(med, precision=0, restart=m, tol=1e-30, maxit=m, max_nrhs=2, no_precond=True)
    u, _ = plan.solve(f)
    for b in range(2):
        ref, size = gmres(p, f[b].astype(CL), m, L, CL)
        assert (abs(u[b] - ref) <= TOL * size).all(), b
