"""The admission footprint counts the work vector of an unpreconditioned or left
step, which a cycle of one complex64 vector does not hold."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def hz():
    from paper_2409_16172_gb300 import build
    build.build()
    from paper_2409_16172_gb300 import hz as _hz
    return _hz


def footprint(hz, restart, **opts):
    o = hz.hz_solver_opts(1, restart, 1e-6, 100, 0, opts.get("no_precond", 0), opts.get("left", 0))
    it = hz.hz_interp(6, 2, 1.0, 0.0, 0.15, 0.0, 0, 0, 0)
    g = hz._grid_of((64, 128))
    return int(hz.lib.hz_request_footprint(C.byref(g), C.byref(it), C.byref(o), 3, 0))


@pytest.mark.parametrize("form", ["no_precond", "left"])
def test_work_vector_of_short_cycles(hz, form):
    n, nrhs = 64 * 128, 3
    assert footprint(hz, 1, **{form: 1}) - footprint(hz, 1) == 8 * n * nrhs
    assert footprint(hz, 2, **{form: 1}) == footprint(hz, 2)
