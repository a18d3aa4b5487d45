"""The operator's integer form (grids of at least 2^17 points) against the FP64
formula in NumPy, element by element: spacings that are equal on all axes and
not, tiles that end inside the grid, periodic edges, damping, both input types,
several right-hand sides; tiles of zeros and of values outside the range of
the integers, NaN and infinity (which reach the neighbours that the formula
gives them to, and nobody else), and media that keep the FP64 form."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def medium(hz, shape, damped, contrast=0.5):
    p = S.small_problem(shape, 3, M=3, Mt=2, width=6, contrast=contrast)
    a = 30.0 * (1.0 + np.random.default_rng(1).random(shape)) if damped else None
    med = hz.Medium(p.c, p.zeta, a, omega=p.omega, M=p.M, Mt=p.Mt, c_o=p.c_o)
    return p, a, med


def formula(p, a, x):
    """(y, magnitude of the terms that are added up at each point)."""
    g = (p.c * (1.0 - 1j * p.zeta)) ** 2
    lap, mag = np.zeros_like(x), np.zeros(x.shape)
    for ax, n in enumerate(p.shape):
        up, dn = np.roll(x, -1, ax), np.roll(x, 1, ax)
        lap += (up - 2 * x + dn) * float(n) ** 2
        mag += (abs(up) + 2 * abs(x) + abs(dn)) * float(n) ** 2
    s = p.omega ** 2 + (0 if a is None else 1j * p.omega * a)
    return g * lap + s * x, abs(g) * mag + abs(s) * abs(x)


def run(hz, med, x, prec):
    import torch
    plan = hz.Plan(med, precision=1, restart=2, max_nrhs=x.shape[0])
    d = torch.from_numpy(x.astype(np.complex64 if prec else np.complex128)).cuda()
    return plan.apply_operator(d).cpu().numpy()


@pytest.mark.parametrize("shape,damped,contrast", [
    ((512, 256), False, 0.5), ((360, 480), True, 0.5), ((2048, 64), False, 0.5), ((720, 720), True, 0.5),
    ((64, 64, 64), False, 0.5), ((60, 48, 96), True, 0.5), ((8, 360, 48), False, 0.5),
    ((512, 512), False, 9.0)])
@pytest.mark.parametrize("prec", [0, 1])
def test_elementwise(shape, damped, contrast, prec):
    hz = hz_module()
    p, a, med = medium(hz, shape, damped, contrast)
    rng = np.random.default_rng(7)
    x = np.stack([S.random_field(rng, shape), S.random_field(rng, shape) * 1e-6])
    if prec:
        x = x.astype(np.complex64).astype(np.complex128)
    y = run(hz, med, x, prec)
    for b in range(2):
        ref, mag = formula(p, a, x[b])
        # sixteen roundings of the terms, and half a unit 2^-56 of the tile's
        # largest value (Gaussian: below 6 standard deviations) in each value
        bound = 16 * EPS * mag + 2.0 ** -56 * abs(x[b]).max() * mag.max() / abs(x[b]).max()
        assert (abs(y[b] - ref) <= bound).all()


@pytest.mark.parametrize("shape", [(512, 256), (64, 64, 64)])
@pytest.mark.parametrize("prec", [0, 1])
def test_special_values(shape, prec):
    hz = hz_module()
    p, a, med = medium(hz, shape, False)
    x = S.random_field(np.random.default_rng(9), shape)[None]
    flat = x.reshape(-1)
    n = flat.size
    x[0, :20] = 0.0                                  # whole tiles of zeros
    x[0, 20:40] *= 1e-30                             # c64: below the integer form's range
    if not prec:
        x[0, 40:50] *= 1e-290
    flat[n // 2 + 5] = complex(np.nan, 1.0)
    flat[3 * n // 4 + 7] = complex(1.0, np.inf)
    if prec:
        x = x.astype(np.complex64).astype(np.complex128)
    y = run(hz, med, x, prec)[0]
    with np.errstate(invalid="ignore"):
        ref, mag = formula(p, a, x[0])
    bad = ~np.isfinite(mag)
    assert 0 < bad.sum() <= 2 * (2 * len(shape) + 1)
    assert (~np.isfinite(y) == bad).all()
    rows = np.abs(np.where(np.isfinite(x[0]), x[0], 0)).max(axis=tuple(range(1, len(shape))))
    near = np.array([np.roll(rows, s) for s in range(-34, 35)]).max(axis=0)
    near = near.reshape((-1,) + (1,) * (len(shape) - 1))  # largest value of any tile with the point
    unit = (mag[~bad].max() / rows.max()) * near * 2.0 ** -56
    assert (abs(y - ref) <= 16 * EPS * mag + unit)[~bad].all()
    assert (y[1:19] == 0).all()


def test_zero_in_zero_out():
    hz = hz_module()
    _, _, med = medium(hz, (512, 256), False)
    assert (run(hz, med, np.zeros((1, 512, 256), np.complex128), 0) == 0).all()
