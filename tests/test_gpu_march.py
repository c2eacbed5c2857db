"""The 3D z-marching operator with planes copied ahead (FP32, odd N + 1, rows of
whole vectors) and without (the same degrees on rows that are not), as a plain
apply and as the operator of the two-launch CG iteration, on single columns
and runs of one and two planes, ragged columns and ragged runs.  Bounds as in
tests/test_gpu_parity.py: 2e-5 for an FP32 apply, 1e-10 for a mixed solve to
1e-13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [(4, 3, 1), (4, 4, 2), (8, 5, 3), (12, 9, 23), (9, 6, 5)])
@pytest.mark.parametrize("N", [0, 2, 4])
def test_march(n, N):
    L = (1.3, 2.1, 0.7)
    o = Oracle(Grid(3, n, L), N, 0.05, 0.6, 0.003)
    h = sdg.Handle(3, n, L, N, 0.05, 0.6, 0.003)
    h.set_profiling()  # every operator launch of a solve by itself, not the resident kernel
    rng = np.random.default_rng(7 * N + n[2])
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    x = rng.standard_normal(o.shape)
    X = dev(x).float()
    Y = torch.empty_like(X)
    h.pressure_apply(X, Y)
    ref = o.pressure_apply(X.cpu().numpy().astype(np.float64))
    assert rel(Y.cpu().numpy(), ref) <= 2e-5
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    h.set_options(sdg.SDG_MIXED, 1e-13, 1e-13, 100000)
    Xs = dev(x0)
    info = h.pressure_cg(dev(b), Xs)
    assert info["status"] == sdg.SDG_OK, info
    assert rel(Xs.cpu().numpy(), o.pressure_solve_exact(b, x0)) <= 1e-10
