"""FP64 operator with the neighbour blocks folded by mirror images (odd N + 1;
in the direct contraction any N >= 2), against the oracle for every degree, on
lines whose values carry a large common offset, and in solves of the degrees
whose accurate contraction is folded.  Bounds as in tests/test_gpu_parity.py:
1e-13 for an FP64 apply (relative to the input where the offset dominates it),
1e-11 for an FP64 solve to 1e-14."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

CASES = [(2, (5, 4), N) for N in range(12)] + [(3, (5, 3, 2), N) for N in range(6)]


def setup(dim, n, N):
    L = (1.3, 2.1, 0.7)[:dim]
    return Oracle(Grid(dim, n, L), N, 0.05, 0.6, 0.003), sdg.Handle(dim, n, L, N, 0.05, 0.6, 0.003)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("dim,n,N", CASES)
def test_fold_apply(dim, n, N):
    o, h = setup(dim, n, N)
    x = np.random.default_rng(40 + N).standard_normal(o.shape)
    for off in (0.0, 1e6):
        X = dev(x + off)
        Y = torch.empty_like(X)
        h.pressure_apply(X, Y)
        y, ref = Y.cpu().numpy(), o.pressure_apply(X.cpu().numpy())
        # A (offset) = 0: the products of the offset round off at 1e-16 of it
        # before they cancel, against 1e-13 for the rest
        assert np.linalg.norm(y - ref) <= 1e-13 * np.linalg.norm(ref) * max(1.0, off)


@pytest.mark.parametrize("dim,n,N", [(2, (5, 4), N) for N in (2, 4, 6, 8)] + [(3, (4, 3, 2), N) for N in (2, 4)])
def test_fold_solve(dim, n, N):
    o, h = setup(dim, n, N)
    rng = np.random.default_rng(60 + N)
    b = o.pressure_apply(rng.standard_normal(o.shape))
    x0 = rng.standard_normal(o.shape)
    h.set_options(sdg.SDG_FP64, 1e-14, 1e-14, 1000000)
    X = dev(x0)
    info = h.pressure_cg(dev(b), X)
    assert info["status"] == sdg.SDG_OK, info
    ex = o.pressure_solve_exact(b, x0)
    assert np.linalg.norm(X.cpu().numpy() - ex) <= 1e-11 * np.linalg.norm(ex)
