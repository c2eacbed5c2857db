"""A wait of the cooperative CG launches that runs out: with a limit of one poll
(no block finds the words of all others at its first look, the others being
still at work) a solve ends with SDG_ERR_CUDA and leaves the handle usable,
whichever kernel waited: the start of a whole resident solve (FP64 and mixed,
2D and 3D), the iterations on small FP32 tiles and on large ones (grids whose
FP64 tiles do not fit, so that the start has no waits).  A grid of one block
waits for nothing.  Solutions afterwards as in tests/test_gpu_resident.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Grid, Oracle  # noqa: E402
from paper_1602_05806_gb300 import sdg  # noqa: E402

F64, MIXED = sdg.SDG_FP64, sdg.SDG_MIXED


@pytest.mark.parametrize("n,N,prec", [((13, 11), 4, F64), ((13, 11), 4, MIXED), ((7, 5, 6), 2, F64), ((7, 5, 6), 2, MIXED),
                                      ((80, 79), 5, MIXED), ((300, 280), 3, MIXED)])
def test_wait_runs_out(n, N, prec):
    L = (6.0, 5.0, 7.0)[:len(n)]
    o = Oracle(Grid(len(n), n, L), N, 0.05, 0.6, 1e-3)
    h = sdg.Handle(len(n), n, L, N, 0.05, 0.6, 1e-3)
    h.set_options(prec, 1e-12, 1e-12, 1000000)
    rng = np.random.default_rng(N)
    b = o.viscous_apply(rng.standard_normal(o.shape))
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    x0 = rng.standard_normal(o.shape)
    for _ in range(2):
        h.set_wait_limit(1)
        with pytest.raises(sdg.SDGError) as e:
            h.viscous_cg(dev(b), dev(x0))
        assert e.value.status == sdg.SDG_ERR_CUDA and "wait" in str(e.value)
        h.set_wait_limit()
        X = dev(x0)
        info = h.viscous_cg(dev(b), X)
        assert info["status"] == sdg.SDG_OK, info
        bound = max(1e-12, 10.0 * max(info["floor_res"], info["eval_res"]))
        assert np.linalg.norm(b - o.viscous_apply(X.cpu().numpy())) <= (1.01 * bound + 1e-13) * np.linalg.norm(b)


def test_one_block_waits_for_nothing():
    o = Oracle(Grid(2, (2, 2), (6.0, 5.0)), 2, 0.05, 0.6, 1e-3)
    h = sdg.Handle(2, (2, 2), (6.0, 5.0), 2, 0.05, 0.6, 1e-3)
    h.set_wait_limit(1)
    b = torch.as_tensor(o.viscous_apply(np.random.default_rng(1).standard_normal(o.shape)), device="cuda")
    assert h.viscous_cg(b, torch.zeros_like(b))["status"] == sdg.SDG_OK


def test_limit_is_checked():
    h = sdg.Handle(2, (2, 2), (1.0, 1.0), 1, 0.1, 0.6, 0.01)
    with pytest.raises(sdg.SDGError) as e:
        h.set_wait_limit(-1)
    assert e.value.status == sdg.SDG_ERR_INVALID_ARG
