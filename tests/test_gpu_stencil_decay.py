"""The operator on fields whose values differ by many orders of magnitude
between neighbouring points, component by component against extended
precision: a bump three cells wide, a wave that decays by 1e-12 within a tile,
a real field with an imaginary part 1e-13 of it, rows that step by 1e-8.  Each
component has to keep the FP64 formula's bound, a few roundings of the
magnitudes of its own terms, on grids that take the integer form (2^17 points
and more) as on smaller ones; and the residual's norm, which the same kernel
forms, the bound that follows."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
L = np.longdouble
FIELDS = ("bump", "decay", "imaginary", "rows")
SHAPES = [((512, 256), False, 0.5), ((360, 480), True, 0.5), ((2048, 64), False, 0.5), ((512, 512), False, 6.0),
          ((64, 64, 64), False, 0.5), ((60, 48, 96), True, 0.5), ((96, 96), True, 0.5)]


def field(name, shape, prec):
    idx = np.indices(shape).astype(float)
    dist = [idx[ax] - 0.4 * n for ax, n in enumerate(shape)]
    x = S.random_field(np.random.default_rng(4), shape)
    if name == "bump":
        x = np.exp(-sum(d * d for d in dist) / 18.0) * (1.0 + 0.3j)
    elif name == "decay":
        x = np.exp(-abs(dist[-1]) + 0.7j * (idx[-1] + idx[0]))
    elif name == "imaginary":
        x = x.real + 1e-13j * x.imag
    else:
        x = x * 1e-8 ** (idx[-2] % 4)
    if prec:
        x = x.astype(np.complex64).astype(np.complex128)
    # no subnormals: not the subject
    x.real[abs(x.real) < (1e-36 if prec else 1e-250)] = 0.0
    x.imag[abs(x.imag) < (1e-36 if prec else 1e-250)] = 0.0
    return x


def problem(hz, shape, damped, contrast):
    p = S.small_problem(shape, 3, M=3, Mt=2, width=6, contrast=contrast)
    a = 30.0 * (1.0 + np.random.default_rng(1).random(shape)) if damped else None
    return p, a, hz.Medium(p.c, p.zeta, a, omega=p.omega, M=p.M, Mt=p.Mt, c_o=p.c_o)


def formula(p, a, x):
    """Real and imaginary part of P x, and the magnitudes of the terms of each."""
    c2, z = p.c.astype(L) ** 2, p.zeta.astype(L)
    gr, gi = c2 * (1 - z * z), -2 * c2 * z
    w2, wa = L(p.omega) ** 2, L(p.omega) * (0 if a is None else a.astype(L))
    lap, mag = [], []
    for v in (x.real.astype(L), x.imag.astype(L)):
        s, m = 0 * v, 0 * v
        for ax, n in enumerate(p.shape):
            up, dn = np.roll(v, -1, ax), np.roll(v, 1, ax)
            s = s + (up - 2 * v + dn) * L(n) ** 2
            m = m + (abs(up) + 2 * abs(v) + abs(dn)) * L(n) ** 2
        lap.append(s)
        mag.append(m)
    xr, xi = x.real.astype(L), x.imag.astype(L)
    re = gr * lap[0] - gi * lap[1] + w2 * xr - wa * xi
    im = gr * lap[1] + gi * lap[0] + w2 * xi + wa * xr
    mre = gr * mag[0] - gi * mag[1] + w2 * abs(xr) + wa * abs(xi)
    mim = gr * mag[1] - gi * mag[0] + w2 * abs(xi) + wa * abs(xr)
    return re, im, mre, mim


@pytest.mark.parametrize("shape,damped,contrast", SHAPES)
@pytest.mark.parametrize("prec", [0, 1])
def test_every_component(shape, damped, contrast, prec):
    import torch
    hz = hz_module()
    p, a, med = problem(hz, shape, damped, contrast)
    plan = hz.Plan(med, precision=1, restart=2, max_nrhs=len(FIELDS))
    x = np.stack([field(name, shape, prec) for name in FIELDS])
    y = plan.apply_operator(torch.from_numpy(x.astype(np.complex64) if prec else x).cuda()).cpu().numpy()
    for b, name in enumerate(FIELDS):
        re, im, mre, mim = formula(p, a, x[b])
        # rounded coefficients (5 eps), and either the FP64 sums (7 eps) or the
        # integer form's values, sums, product and conversion (11 eps)
        assert (abs(y[b].real - re) <= 16 * EPS * mre).all(), name
        assert (abs(y[b].imag - im) <= 16 * EPS * mim).all(), name


@pytest.mark.parametrize("shape,damped,contrast", SHAPES)
def test_residual_norm(shape, damped, contrast):
    hz = hz_module()
    p, a, med = problem(hz, shape, damped, contrast)
    plan = hz.Plan(med, precision=1, restart=2, tol=1e30, max_nrhs=len(FIELDS))
    u = np.stack([field(name, shape, 0) for name in FIELDS])
    f = np.stack([S.random_field(np.random.default_rng(6 + b), shape) * 1e3 for b in range(len(FIELDS))])
    _, stats = plan.solve(f, u.copy())  # the tolerance is met at once
    for b, name in enumerate(FIELDS):
        re, im, mre, mim = formula(p, a, u[b])
        rr, ri = f[b].real - re, f[b].imag - im
        norm = np.sqrt((rr * rr + ri * ri).sum())
        nf = np.linalg.norm(f[b])
        bound = 17 * EPS * np.sqrt((mre * mre + mim * mim).sum()) + 64 * EPS * norm
        assert stats[b]["iters"] == 0
        assert abs(stats[b]["rel_true_resid"] * nf - norm) <= bound, name
