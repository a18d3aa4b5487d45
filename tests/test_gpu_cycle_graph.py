"""Cycles captured as a graph only after a plan's first full cycles: solves of
more cycles than that, of fewer, and of another right-hand-side count on the
same plan give bit for bit what direct launches give."""
import numpy as np
import pytest

from paper_2409_16172_gb300 import synth as S

from gpu_util import hz_module, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("restart", [2, 7])
def test_captured_cycles_equal_direct_ones(precision, restart):
    hz = hz_module()
    p = S.small_problem((48, 64), 5, M=5, Mt=3, width=4)
    med, _ = media(hz, p, oracle=False)
    rng = np.random.default_rng(2)
    f = np.stack([S.random_field(rng, p.shape) for _ in range(3)])
    direct = hz.Plan(med, precision=precision, restart=restart, tol=1e-9, maxit=60, max_nrhs=3)
    graph = hz.Plan(med, precision=precision, restart=restart, tol=1e-9, maxit=60, max_nrhs=3,
                    graphs=True)
    for nrhs in (1, 3, 1, 2, 2):
        a, sa = direct.solve(f[:nrhs])
        b, sb = graph.solve(f[:nrhs])
        assert np.array_equal(a, b)
        assert [s["iters"] for s in sa] == [s["iters"] for s in sb]
    assert sa[0]["restarts"] > 4
