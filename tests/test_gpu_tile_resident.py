"""Operator shapes and the cooperative CG launches: a tuned shape never moves a
solve away from them, a shape asked for moves only solves of a precision that
has it (2D: FP32 iterations, 3D: both).  A solve with cooperative launches
counts fewer kernels than iterations, the two-launch form two per iteration."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402


def setup(n, N):
    L = (6.0, 5.0, 7.0)[:len(n)]
    o = Oracle(Grid(len(n), n, L), N, 0.05, 0.6, 0.03)
    h = sdg.Handle(len(n), n, L, N, 0.05, 0.6, 0.03)
    b = torch.as_tensor(o.pressure_apply(np.random.default_rng(N).standard_normal(o.shape)), device="cuda")
    return h, b


def cooperative(h, b, prec):
    h.set_options(prec, 1e-12, 1e-12, 1000000)
    before = h.counters()["launches"]
    info = h.pressure_cg(b, torch.zeros_like(b))
    launches = h.counters()["launches"] - before
    assert info["status"] == sdg.SDG_OK and info["iters"] >= 40, info
    assert launches < info["iters"] or launches >= 2 * info["iters"]
    return launches < info["iters"]


@pytest.mark.parametrize("n,N", [((16, 16), 4), ((33, 20), 3), ((64, 64), 5), ((24, 31), 7), ((8, 6, 7), 4), ((9, 9, 9), 2)])
def test_tuned_shape(n, N):
    h, b = setup(n, N)
    for _ in range(3):
        h.autotune()
        assert cooperative(h, b, sdg.SDG_FP64)
        assert cooperative(h, b, sdg.SDG_MIXED)


@pytest.mark.parametrize("n,N", [((16, 16), 4), ((8, 6, 7), 3)])
def test_shape_asked_for(n, N):
    h, b = setup(n, N)
    for v in (1, 2):
        h.set_tile(v)
        assert cooperative(h, b, sdg.SDG_FP64) == (len(n) == 2)
        assert not cooperative(h, b, sdg.SDG_MIXED)
    h.set_tile(0)
    assert cooperative(h, b, sdg.SDG_MIXED)
