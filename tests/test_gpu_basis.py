"""The Gram-Schmidt kernels on the block fixed-point basis: Hessenberg columns
of one unpreconditioned Arnoldi cycle against an Arnoldi process (CGS2, FP64)
written here with the oracle's operator, at sizes around the kernels' edges:
grids of less than one tile of 128 points, of whole tiles and of a tile and a
bit, cycles across the fused kernel's ring sizes (24, 34 and 52 rows) and its
limit of 44 vectors, one to 128 vectors, several right-hand sides of very
different size."""
import numpy as np
import pytest

import oracle as O
from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module

pytestmark = pytest.mark.gpu

# FP64 Arnoldi columns of these cases move by at most 2.7e-15 of the largest
# entry when f is perturbed by 1e-15 relative (four perturbations each, the
# NumPy process below): rounding of a few 1e-16 per operation stays far below
TOL = 1e-12
CASES = [((8, 8), 1, 1), ((8, 8), 6, 2), ((12, 12), 16, 1), ((16, 24), 17, 3), ((24, 20), 24, 1),
         ((24, 20), 25, 2), ((8, 12, 16), 36, 1), ((48, 48), 46, 1), ((48, 64), 64, 1), ((64, 96), 128, 2)]


def arnoldi(apply_op, f, m):
    n = f.size
    V = np.zeros((m + 1, n), np.complex128)
    H = np.zeros((m + 1, m), np.complex128)
    V[0] = f.ravel() / np.linalg.norm(f)
    for j in range(m):
        w = apply_op(V[j].reshape(f.shape)).ravel()
        for _ in range(2):
            h = V[:j + 1].conj() @ w
            w = w - V[:j + 1].T @ h
            H[:j + 1, j] += h
        H[j + 1, j] = np.linalg.norm(w)
        V[j + 1] = w / H[j + 1, j]
    return H


def problem(shape, nrhs):
    p = S.small_problem(shape, 11, M=3, Mt=2, width=2)
    rng = np.random.default_rng(5)
    f = np.stack([S.random_field(rng, shape) * 1e3 ** (b - 1) for b in range(nrhs)])
    return p, f


@pytest.mark.parametrize("shape,m,nrhs", CASES)
def test_hessenberg_columns(shape, m, nrhs):
    hz = hz_module()
    p, f = problem(shape, nrhs)
    med = hz.Medium(p.c, p.zeta, omega=p.omega, M=p.M, Mt=p.Mt, c_o=p.c_o)
    med_o = O.make_medium(p.c, p.zeta, None, p.omega, p.M, p.Mt, p.c_o, None, 0.15)
    plan = hz.Plan(med, precision=0, restart=m, tol=1e-30, maxit=m, max_nrhs=nrhs, no_precond=True)
    plan.solve(f)
    for b in range(nrhs):
        H = plan.hessenberg(b)
        ref = arnoldi(lambda x: O.apply_operator(med_o, x), f[b], m)
        assert H.shape == ref.shape
        assert np.abs(H - ref).max() <= TOL * np.abs(ref).max(), b
