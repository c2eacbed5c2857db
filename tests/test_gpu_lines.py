"""The line-wise stage kernels (projections, divergence, velocity update,
convection) for every degree in 2D and 3D, on grids whose rows end inside a
run of elements, and on single cells (both neighbours are the cell itself).
Bound as for the stages in tests/test_gpu_parity.py: 1e-13 (a handful of
roundings per output).  The convection's time step keeps each sub-step at a
tenth of the CFL limit: rough data near the limit grow, and their roundings
with them."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

CASES = ([(2, (67, 3) if N < 3 else (35, 4), N) for N in range(12)] + [(2, (1, 1), 3), (2, (1, 41), 6)]
         + [(3, (9, 2, 3) if N < 6 else (3, 1, 2), N) for N in range(12)] + [(3, (1, 13, 1), 4)])


def rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


@pytest.mark.parametrize("theta", [0.6, 1.0])
@pytest.mark.parametrize("dim,n,N", CASES)
def test_line_stages(dim, n, N, theta):
    L = (1.3, 2.1, 0.7)[:dim]
    o = Oracle(Grid(dim, n, L), N, 0.05, theta, 0.003)
    h = sdg.Handle(dim, n, L, N, 0.05, theta, 0.003)
    rng = np.random.default_rng(100 + N)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    host = lambda t: t.cpu().numpy()
    U = [rng.standard_normal(o.shape) for _ in range(dim)]
    P0, P1 = rng.standard_normal(o.shape), rng.standard_normal(o.shape)
    D = [dev(u) for u in U]
    out = [torch.empty_like(D[0]) for _ in range(dim)]
    for d in range(dim):
        h.dual_to_main(d, D[d], out[d])
        assert rel(host(out[d]), o.dual_to_main(U[d], d)) <= 1e-13
        h.main_to_dual(d, D[d], out[d])
        assert rel(host(out[d]), o.main_to_dual(U[d], d)) <= 1e-13
    b = torch.empty_like(D[0])
    h.pressure_rhs(D, dev(P0), b)
    ref = o.pressure_rhs(U, P0)
    # (relative to the terms that cancel in b where it is small)
    assert np.linalg.norm(host(b) - (ref - ref.mean())) <= 1e-13 * (np.linalg.norm(ref) + 1e-3)
    h.velocity_update(D, dev(P1), dev(P0), out)
    for d, r in enumerate(o.velocity_update(U, theta * P1 + (1 - theta) * P0)):
        assert rel(host(out[d]), r) <= 1e-13
    V = [0.1 * u for u in U]
    cfl = 0.003 * (2 * N + 1) * sum(np.abs(V[d]).max() * n[d] / L[d] for d in range(dim))
    o.nsub = max(2, math.ceil(cfl / 0.1))
    h.set_convection_substeps(o.nsub)
    h.convect([dev(v) for v in V], out)
    for d, r in enumerate(o.rk3(V)):
        assert rel(host(out[d]), r) <= 1e-13
