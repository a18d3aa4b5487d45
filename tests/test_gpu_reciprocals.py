"""The FP64 reciprocal and reciprocal square root of csrc/recip.cuh against
extended precision: a probe compiled from the header, on values over the whole
range of exponents whose reciprocal is normal and on all mantissas' leading
bits.  Bounds: the final rounding (2^-53 of the result, at most), for the
square root also the rounding of x y (2^-53 in e, half of it in the result),
and a tenth or a quarter of 2^-53 for the terms left out and second-order
roundings."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = """
#include "recip.cuh"
__global__ void k(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = hz::recip3(x[i]);
    s[i] = hz::rsqrt3(x[i]);
  }
}
extern "C" int probe(const void* x, void* r, void* s, int n) {
  k<<<(n + 255) / 256, 256>>>((const double*)x, (double*)r, (double*)s, n);
  return cudaDeviceSynchronize();
}
"""


def test_within_the_stated_bounds(tmp_path):
    import torch
    from paper_2409_16172_gb300 import build
    src, lib = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text(PROBE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", str(lib), str(src)],
                   check=True)
    rng = np.random.default_rng(3)
    mant = np.concatenate([1.0 + np.arange(1 << 16) / float(1 << 16), 1.0 + rng.random(1 << 17),
                           2.0 - 2.0 ** -52 * np.arange(1, 64), 1.0 + 2.0 ** -52 * np.arange(64)])
    x = np.ldexp(mant, rng.integers(-1021, 1021, mant.size))
    d = torch.from_numpy(x).cuda()
    r, s = torch.empty_like(d), torch.empty_like(d)
    p = ctypes.c_void_p
    assert ctypes.CDLL(str(lib)).probe(p(d.data_ptr()), p(r.data_ptr()), p(s.data_ptr()), x.size) == 0
    q = x.astype(np.longdouble)
    assert np.finfo(np.longdouble).nmant >= 63
    er = abs(r.cpu().numpy() * q - 1)
    es = abs(s.cpu().numpy() * np.sqrt(q) - 1)
    assert er.max() <= 1.1 * 2.0 ** -53, float(er.max())
    assert es.max() <= 1.75 * 2.0 ** -53, float(es.max())
