"""The complex128 apply is as accurate as one with FP64 transforms: its error
against extended precision, for noise and for inputs whose spectra or values
span many orders of magnitude, beside the oracle's (NumPy's complex128
transforms, symbol and weights in FP64) on the same inputs.  In the 2-norm at
most 1.6 times that (another order of the same roundings); for smooth inputs,
whose spectrum is a few large entries, also in the maximum norm, at most twice."""
import numpy as np
import pytest

import oracle as O
from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu

L, CL = np.longdouble, np.clongdouble
SMOOTH = ("bump", "wide", "plane")


def inputs(shape):
    idx = np.indices(shape).astype(float)
    noise = S.random_field(np.random.default_rng(5), shape)
    r2 = sum((idx[a] - shape[a] * 0.45) ** 2 for a in range(len(shape)))
    point = np.zeros(shape, complex)
    point[tuple(s // 3 for s in shape)] = 1.0
    return {"noise": noise, "rows": noise * 10.0 ** -(idx[-2] % 8), "cols": noise * 10.0 ** -(idx[-1] % 8),
            "point": point, "bump": np.exp(-r2 / 18.0) * (1 + 0.3j), "wide": np.exp(-r2 / 540.0) * (1 + 0.3j),
            "plane": np.exp(2j * np.pi * (3 * idx[-1] / shape[-1] + 5 * idx[-2] / shape[-2]))}


def setup(p, info):
    """Symbols q_k and hat weights w_k in extended precision, from the nodes and
    interpolation parameters as the library holds them in FP64."""
    xi2 = np.zeros(p.shape, L)
    for a, n in enumerate(p.shape):
        k = np.arange(n)
        x = 2.0 * np.pi * np.where(k <= (n - 1) // 2, k, k - n)
        b = [1] * len(p.shape)
        b[a] = n
        xi2 = xi2 + (x * x).astype(L).reshape(b)
    gam, ak, M, Mt = info["gamma"], info["a"], p.M, p.Mt
    q = [1 / (CL(complex(p.omega * p.omega, p.omega * ak[k]))
              - CL(complex(g.real * g.real - g.imag * g.imag, 2 * g.real * g.imag)) * xi2)
         for k, g in enumerate(gam)]
    w = [np.zeros(p.shape, L) for _ in gam]

    def hats(value, nodes, seg0, index, where):
        m = np.clip(np.searchsorted(nodes, value, side="right") - 1, 0, len(nodes) - 2)
        t = np.clip((value - nodes[m]) / (nodes[m + 1] - nodes[m]), 0.0, 1.0)
        t = ((seg0 + m) + t) - (seg0 + m)  # as a segment number and its fraction
        for i in range(len(nodes) - 1):
            s = (m == i) & where
            w[index[i]][s] += 1 - t[s].astype(L)
            w[index[i + 1]][s] += t[s].astype(L)

    layer = p.zeta > 0
    hats(p.c, gam[:M].real, 0, range(M), ~layer)
    if Mt:
        co = int(np.where(gam[:M].real == p.c_o)[0][0])
        hats(p.zeta, p.zeta.max() * np.arange(Mt + 1) / Mt, M, [co, *range(M, M + Mt)], layer)
    return q, w


def apply_q(q, w, x):
    xh = np.fft.fftn(x)
    return sum(wk * np.fft.ifftn(qk * xh) for qk, wk in zip(q, w))


@pytest.mark.parametrize("shape,M,Mt", [((120, 180), 6, 0), ((128, 128), 5, 2), ((40, 48, 60), 4, 2)])
def test_as_accurate_as_fp64_transforms(shape, M, Mt):
    import torch
    hz = hz_module()
    p = S.small_problem(shape, 3, M=M, Mt=Mt, width=8 if Mt else 0, ppw=8.0)
    med, med_o = media(hz, p)
    plan = hz.Plan(med, precision=0, restart=2)
    q, w = setup(p, med.info())
    for name, x in inputs(shape).items():
        ref = apply_q(q, w, x.astype(CL))
        e_o = abs(O.apply_preconditioner(med_o, x) - ref)
        e = abs(plan.apply_preconditioner(torch.from_numpy(x).cuda(), precision=0).cpu().numpy() - ref)
        two, two_o = np.sqrt((e ** 2).sum()), np.sqrt((e_o ** 2).sum())
        assert two <= 1.6 * two_o, (name, float(two / two_o))
        if name in SMOOTH:
            assert e.max() <= 2.0 * e_o.max(), (name, float(e.max() / e_o.max()))
