"""The resident CG (one cooperative launch per segment of iterations, tiles of
the grid in registers and shared memory) at the edges of its tiling: single
cells and single tiles (neighbours wrap inside the tile), ragged last tiles,
every parity of the degree, two lines per thread, grids near its capacity,
both precisions and both systems.

Bounds: a solve ends with a true residual of at most max(rtol, 3 floor), or
ten times the floor once it stalls (include/sdg.h); the oracle evaluates A x
with another rounding, of at most a few floors for N <= 9 (for N = 11 it is 1e-14
by itself, so there only the library's own residual counts), hence the factor
1.5.  On
small grids up to N = 6 the solution is compared with the oracle's exact one at
the bounds and the rtol (1e-14) of tests/test_gpu_parity.py: 1e-11 FP64, 1e-10
mixed, ten times those for the pressure of odd degrees (near-kernel modes)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle, cg  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

TWO_PI = 2.0 * math.pi

CASES = [
    (2, (1, 1), 3), (2, (1, 7), 2), (2, (2, 2), 7), (2, (3, 33), 0), (2, (5, 9), 1), (2, (13, 11), 4),
    (2, (9, 14), 6), (2, (11, 5), 9), (2, (7, 6), 11), (2, (80, 79), 5), (2, (128, 81), 7),
    (3, (1, 1, 1), 2), (3, (2, 1, 5), 3), (3, (5, 4, 3), 0), (3, (7, 5, 6), 1), (3, (4, 6, 5), 4), (3, (5, 3, 4), 5),
    (3, (13, 12, 11), 3),
]


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def host(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy()


@pytest.mark.parametrize("prec", [sdg.SDG_FP64, sdg.SDG_MIXED])
@pytest.mark.parametrize("dim,n,N", CASES)
def test_resident_solves(dim, n, N, prec):
    L = (TWO_PI, 0.8 * TWO_PI, 1.3 * TWO_PI)[:dim]
    o = Oracle(Grid(dim, n, L), N, 0.05, 0.6, 0.03)
    h = sdg.Handle(dim, n, L, N, 0.05, 0.6, 0.03)
    h.set_options(prec, 1e-14, 1e-14, 1000000)
    rng = np.random.default_rng(7 + N)
    tol = 1e-11 if prec == sdg.SDG_FP64 else 1e-10
    small = math.prod(n) <= 200
    for A, solve, exact in ((o.pressure_apply, h.pressure_cg, o.pressure_solve_exact),
                            (o.viscous_apply, h.viscous_cg, lambda b, x0: o.viscous_solve_exact(b))):
        b = A(rng.standard_normal(o.shape))
        x0 = rng.standard_normal(o.shape)
        before = h.counters()["launches"]
        X = dev(x0)
        info = solve(dev(b), X)
        assert info["status"] == sdg.SDG_OK, info
        bound = max(1e-14, 10.0 * max(info["floor_res"], info["eval_res"]))
        assert info["true_res"] <= bound, info
        # fewer launches than iterations: the resident kernel ran (FP64 tiles
        # of the two largest grids do not fit)
        if info["iters"] >= 64 and (prec == sdg.SDG_MIXED or small):
            assert h.counters()["launches"] - before < info["iters"]
        x = host(X)
        nb = np.linalg.norm(b)
        if nb == 0.0:
            continue
        assert N > 9 or np.linalg.norm(b - A(x)) <= 1.5 * bound * nb
        if small and N <= 6:
            ex = exact(b, x0)
            odd = 10.0 if N % 2 and A == o.pressure_apply else 1.0
            assert np.linalg.norm(x - ex) <= odd * tol * np.linalg.norm(ex)


@pytest.mark.parametrize("dim,n,N", [(2, (9, 6), 3), (3, (4, 5, 3), 2)])
def test_resident_stops_at_maxit(dim, n, N):
    """A capped mixed solve returns the iterate of plain CG (its last step
    included) at FP32 accuracy, and a start vector that already solves the
    system comes back unchanged."""
    L = (TWO_PI,) * dim
    o = Oracle(Grid(dim, n, L), N, 0.05, 0.6, 0.03)
    h = sdg.Handle(dim, n, L, N, 0.05, 0.6, 0.03)
    rng = np.random.default_rng(3)
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    for prec, tol in ((sdg.SDG_FP64, 1e-12), (sdg.SDG_MIXED, 1e-5)):
        h.set_options(prec, 1e-14, 1e-14, 4)
        X = dev(x0)
        info = h.pressure_cg(dev(b), X, ok=(sdg.SDG_OK, sdg.SDG_ERR_NOT_CONVERGED))
        # (a mixed solve that pauses for a replacement at the cap makes one more iteration)
        assert info["status"] == sdg.SDG_ERR_NOT_CONVERGED
        assert info["iters"] == 4 or (prec == sdg.SDG_MIXED and info["iters"] == 5)
        ref = cg(o.pressure_apply, b, x0, 1e-30, maxit=info["iters"]).x
        # (four FP32 iterations of a residual of order ||b||: 2^-24 times a few tens)
        assert np.linalg.norm(host(X) - ref) <= tol * np.linalg.norm(ref)
        Z = dev(x0)
        info = h.pressure_cg(dev(np.zeros_like(b)), Z, ok=(sdg.SDG_OK, sdg.SDG_ERR_NOT_CONVERGED))
        assert info["status"] == sdg.SDG_OK and info["iters"] == 0
        assert np.linalg.norm(host(Z) - x0) <= 1e-13 * np.linalg.norm(x0)


# grids above one or two lines per thread: large tiles with an odd number of
# elements, ragged last tiles, one and several rounds past the registers
LARGE = [((512, 430), 0), ((268, 289), 1), ((300, 290), 2), ((300, 280), 3), ((225, 211), 4), ((119, 257), 5),
         ((150, 171), 6), ((256, 256), 7), ((160, 150), 7), ((274, 116), 8), ((255, 79), 9), ((110, 120), 10), ((128, 128), 11)]


@pytest.mark.parametrize("n,N", LARGE)
def test_resident_large_tiles(n, N):
    """Mixed solves on large 2D tiles: the viscous system to 1e-12 and the
    pressure system to 1e-3, whose FP32 iterations the FP64 residual confirms;
    residuals evaluated by the oracle (its rounding: below 1e-13)."""
    L = (TWO_PI, 1.2 * TWO_PI)
    o = Oracle(Grid(2, n, L), N, 0.05, 0.6, 1e-3)
    h = sdg.Handle(2, n, L, N, 0.05, 0.6, 1e-3)
    rng = np.random.default_rng(N)
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    for A, solve, rtol in ((o.viscous_apply, h.viscous_cg, 1e-12), (o.pressure_apply, h.pressure_cg, 1e-3)):
        h.set_options(sdg.SDG_MIXED, rtol, rtol, 1000000)
        before = h.counters()["launches"]
        X = dev(x0)
        info = solve(dev(b), X)
        assert info["status"] == sdg.SDG_OK, info
        bound = max(rtol, 10.0 * max(info["floor_res"], info["eval_res"]))
        assert np.linalg.norm(b - A(host(X))) <= (1.01 * bound + 1e-13) * np.linalg.norm(b)
        # far fewer launches than two per iteration: the resident kernel ran
        assert info["iters"] < 64 or h.counters()["launches"] - before < info["iters"]
