"""The two-launch CG iteration on grids whose tiles do not fit the cooperative
kernels (the default there), and on small ones with form 1: FP64 with every
parity of the degree (folded and even/odd contraction, operators of less than a
wave of blocks spread over the SMs by their shared memory), FP32 beyond the
large tiles.  Two launches per iteration are counted.  Bounds as in
tests/test_gpu_resident.py (oracle-side residual) and tests/test_gpu_parity.py
(1e-11 FP64, ten times that for the pressure of odd degrees, 1e-10 mixed, for
solutions to 1e-14; 1e-12 for capped FP64 iterates)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle, cg  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

F64, MIXED = sdg.SDG_FP64, sdg.SDG_MIXED


def setup(n, N):
    L = (6.0, 5.0, 7.0)[:len(n)]
    return Oracle(Grid(len(n), n, L), N, 0.05, 0.6, 1e-3), sdg.Handle(len(n), n, L, N, 0.05, 0.6, 1e-3)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def norm(a):
    return np.linalg.norm(a)


LARGE = [((100, 90), 6, F64), ((180, 170), 2, F64), ((200, 190), 1, F64), ((90, 60), 9, F64), ((80, 70), 8, F64),
         ((130, 120), 4, F64), ((30, 24, 27), 3, F64), ((24, 22, 20), 4, F64), ((21, 20, 20), 2, F64), ((280, 270), 7, MIXED),
         ((32, 26, 24), 4, MIXED), ((47, 45, 21), 3, MIXED)]


@pytest.mark.parametrize("n,N,prec", LARGE)
def test_large_grids(n, N, prec):
    o, h = setup(n, N)
    rng = np.random.default_rng(N)
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    for A, solve, rtol in ((o.viscous_apply, h.viscous_cg, 1e-12), (o.pressure_apply, h.pressure_cg, 1e-3)):
        h.set_options(prec, rtol, rtol, 1000000)
        before = h.counters()["launches"]
        X = dev(x0)
        info = solve(dev(b), X)
        assert info["status"] == sdg.SDG_OK, info
        assert h.counters()["launches"] - before >= 2 * info["iters"] > 0
        bound = max(rtol, 10.0 * max(info["floor_res"], info["eval_res"]))
        assert norm(b - A(X.cpu().numpy())) <= (1.01 * bound + 1e-13) * norm(b)
    if prec == F64:  # x as plain CG leaves it after three iterations
        h.set_options(F64, 1e-14, 1e-14, 3)
        X = dev(x0)
        info = h.pressure_cg(dev(b), X, ok=(sdg.SDG_ERR_NOT_CONVERGED,))
        ref = cg(o.pressure_apply, b, x0, 1e-30, maxit=3).x
        assert info["iters"] == 3 and norm(X.cpu().numpy() - ref) <= 1e-12 * norm(ref)


SMALL = [((5, 4), N) for N in range(7)] + [((12, 11), 8), ((1, 6), 4), ((5, 4, 3), 1), ((5, 4, 3), 2), ((4, 3, 2), 4)]


@pytest.mark.parametrize("prec", [F64, MIXED])
@pytest.mark.parametrize("n,N", SMALL)
def test_small_grids(n, N, prec):
    o, h = setup(n, N)
    h.set_iteration_form(1)
    h.set_options(prec, 1e-14, 1e-14, 1000000)
    rng = np.random.default_rng(60 + N)
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    before = h.counters()["launches"]
    X = dev(x0)
    info = h.pressure_cg(dev(b), X)
    assert info["status"] == sdg.SDG_OK, info
    assert h.counters()["launches"] - before >= 2 * info["iters"]
    bound = max(1e-14, 10.0 * max(info["floor_res"], info["eval_res"]))
    assert norm(b - o.pressure_apply(X.cpu().numpy())) <= 1.5 * bound * norm(b)
    if N <= 6:
        ex = o.pressure_solve_exact(b, x0)
        assert norm(X.cpu().numpy() - ex) <= (1e-11 if prec == F64 else 1e-10) * (10.0 if N % 2 else 1.0) * norm(ex)


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("n,N", [((7, 5), N) for N in range(12)] + [((5, 4, 3), N) for N in range(6)])
def test_offset_in_the_accurate_contraction(n, N, form):
    """A start vector that solves the system but for a constant of 1e6 (the
    kernel of the operator): its residual, formed with the accurate contraction
    by the launches (form 1) or the cooperative kernel (2), is that of an FP64
    apply without the offset (1e-13, and as much for the oracle's b; an offset
    that reached the products would leave 1e-10)."""
    o, h = setup(n, N)
    h.set_iteration_form(form)
    x = np.random.default_rng(80 + N).standard_normal(o.shape) + 1e6
    b = o.pressure_apply(x - 1e6)  # (the difference is exact)
    X = dev(x)
    info = h.pressure_cg(dev(b), X)
    assert info["status"] == sdg.SDG_OK and info["iters"] == 0, info
    assert info["true_res"] <= 2e-13, info
