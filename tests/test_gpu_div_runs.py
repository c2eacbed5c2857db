"""The divergence by runs of elements and the velocity update of all directions
in one launch: grids with fewer elements in a run than a block holds, ragged
last runs, more runs than blocks (every block takes several), an update in
place.  Bounds as in tests/test_gpu_lines.py (1e-13)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

CASES = [((31, 21), 8), ((13, 12), 0), ((2, 3), 5), ((64, 63), 3), ((240, 230), 5), ((5, 7, 3), 2), ((1, 2, 1), 7), ((24, 24, 24), 4),
         ((11, 11, 11), 11)]


@pytest.mark.parametrize("n,N", CASES)
def test_divergence_and_update(n, N):
    dim = len(n)
    L = (1.3, 2.1, 0.7)[:dim]
    o = Oracle(Grid(dim, n, L), N, 0.05, 0.6, 0.003)
    h = sdg.Handle(dim, n, L, N, 0.05, 0.6, 0.003)
    rng = np.random.default_rng(N)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    U = [rng.standard_normal(o.shape) for _ in range(dim)]
    P0, P1 = rng.standard_normal(o.shape), rng.standard_normal(o.shape)
    D = [dev(u) for u in U]
    b = torch.empty_like(D[0])
    for _ in range(2):  # (the ticket of the sum is ready for the next launch)
        h.pressure_rhs(D, dev(P0), b)
        ref = o.pressure_rhs(U, P0)
        assert np.linalg.norm(b.cpu().numpy() - (ref - ref.mean())) <= 1e-13 * (np.linalg.norm(ref) + 1e-3)
    h.velocity_update(D, dev(P1), dev(P0), D)
    for d, r in enumerate(o.velocity_update(U, 0.6 * P1 + 0.4 * P0)):
        assert np.linalg.norm(D[d].cpu().numpy() - r) <= 1e-13 * np.linalg.norm(r)
