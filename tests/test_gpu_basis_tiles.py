"""The Gram-Schmidt kernels on the block fixed-point basis of a preconditioned
solve: Hessenberg columns of one complex128 cycle against an Arnoldi process
(CGS2, FP64) written here with the oracle's operator and preconditioner.  Small
grids, of less than a tile of 128 points, whole tiles, and a tile and a bit,
with one vector to 128; and grids of more tiles than the kernels have blocks
(608), where a block walks over several, its last one partial: cycles across the
fused kernel's ring sizes (24, 34 and 52 rows), its limit of 44 vectors and past
it, one right-hand side and three of very different size."""
import numpy as np
import pytest

import oracle as O
from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu

# FP64 Arnoldi columns of these cases move by at most 1.2e-14 of the largest
# entry when every operator result is perturbed by 1e-15 relative (two
# perturbations each of six cases, the process below)
TOL = 1e-12


def arnoldi(apply_op, f, m):
    V = np.zeros((m + 1, f.size), np.complex128)
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


@pytest.mark.parametrize("shape,m,nrhs", [
    ((8, 8), 1, 1), ((8, 8), 6, 2), ((12, 12), 16, 1), ((16, 24), 17, 3), ((24, 20), 24, 1), ((24, 20), 25, 2),
    ((8, 12, 16), 36, 1), ((48, 48), 46, 1), ((48, 64), 64, 1), ((64, 96), 128, 2),
    ((360, 360), 26, 3), ((360, 360), 64, 1), ((60, 48, 40), 46, 1), ((512, 512), 38, 1)])
def test_hessenberg_columns(shape, m, nrhs):
    hz = hz_module()
    p = S.small_problem(shape, 11, M=3, Mt=2, width=12 if max(shape) > 300 else 2)
    rng = np.random.default_rng(5)
    f = np.stack([S.random_field(rng, shape) * 1e3 ** (b - 1) for b in range(nrhs)])
    med, med_o = media(hz, p)
    plan = hz.Plan(med, precision=0, restart=m, tol=1e-30, maxit=m, max_nrhs=nrhs)
    plan.solve(f)
    for b in range(nrhs):
        H = plan.hessenberg(b)
        ref = arnoldi(lambda v: O.apply_operator(med_o, O.apply_preconditioner(med_o, v)), f[b], m)
        assert H.shape == ref.shape
        assert np.abs(H - ref).max() <= TOL * np.abs(ref).max(), b
