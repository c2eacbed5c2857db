"""The projections of degree 1 against extended precision: no further from it
than the same sums formed term by term in FP64, within a tenth (the scatter of
such errors over 20,000 values is a few percent; the even/odd form, with two
more roundings per term, would be at 1.2 to 1.5 times)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_05806_gb300 import sdg  # noqa: E402


def transform(R, L, x, s, axis, shift_r, shift_l, dtype):
    """R x[e + shift_r] + s L x[e + shift_l] along an axis of nodes, term by term."""
    ex = x.ndim // 2 - (x.ndim - axis)
    a = np.moveaxis(np.roll(x, -shift_r, ex), axis, -1).astype(dtype)
    b = np.moveaxis(np.roll(x, -shift_l, ex), axis, -1).astype(dtype)
    out = np.zeros_like(a)
    wide = np.longdouble
    for m in range(2):
        for q in range(2):  # (one rounding per multiply-add)
            for c, v in ((R[m, q], a), (s * L[m, q], b)):
                out[..., m] = (wide(c) * v[..., q].astype(wide) + out[..., m]).astype(dtype)
    return out


@pytest.mark.parametrize("n", [(71, 70), (16, 14, 12)])
def test_degree_one(n):
    dim, LD = len(n), np.longdouble
    L = (2.0 * np.pi,) * dim
    h = sdg.Handle(dim, n, L, 1, 0.05, 0.6, 0.003)
    M, w = sdg.sdg_matrices(1), sdg.sdg_nodes(1)[1]
    # the exact matrices: nodes (1 -+ 1 / sqrt 3) / 2, weights 1/2, quadrature exact for the cubic integrands
    r3 = np.sqrt(LD(3))
    xi = np.array([(1 - 1 / r3) / 2, (1 + 1 / r3) / 2])
    phi = lambda x: np.array([(x - xi[1]) / (xi[0] - xi[1]), (x - xi[0]) / (xi[1] - xi[0])])
    lo, hi = phi(xi / 2), phi((xi + 1) / 2)
    ML, MR = (lo @ hi.T) / 4, (hi @ lo.T) / 4
    rng = np.random.default_rng(5)
    x = rng.standard_normal(h.shape)
    X = torch.as_tensor(x, device="cuda")
    Y = torch.empty_like(X)
    err = lambda y, e: float(np.sqrt((((y - e) / np.sqrt((e * e).sum())) ** 2).sum()))
    for d in range(dim):
        axis = 2 * dim - 1 - d
        for f, sr, sl in ((h.dual_to_main, 0, -1), (h.main_to_dual, 1, 0)):
            f(d, X, Y)
            got = np.moveaxis(Y.cpu().numpy(), axis, -1)
            exact = 2 * transform(MR, ML, x, 1, axis, sr, sl, LD)
            plain = transform(M["MR"], M["ML"], x, 1, axis, sr, sl, np.float64) * (1.0 / w)
            assert err(got, exact) <= 1.1 * err(plain, exact), (d, err(got, exact) / err(plain, exact))
