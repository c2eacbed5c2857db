"""A solve whose cooperative launch the GPU refuses (as where the stream's
context has fewer SMs than the device) runs with launches per iteration
instead.  The refusal is made by a stand-in for the runtime's launch call
(tests/fake_cudart.c): on the CPU with kernels that do nothing, so that such a
solve ends at the host's cap on batches, and on the GPU with real ones."""
import pytest

from paper_1602_05806_gb300 import build
from tests import fake_runtime

# start of a whole resident solve, FP32 iterations on small and on large tiles
GRIDS = [((13, 11), 4), ((7, 5, 6), 2), ((80, 79), 5), ((120, 110), 3)]

CPU = """
import ctypes
from paper_1602_05806_gb300 import sdg
h = sdg.Handle({dim}, {n}, (1.0,) * 3, {N}, 0.1, 0.6, 0.01)
x, y = (ctypes.create_string_buffer(8 * h.ndof) for _ in range(2))
for prec in (0, 1):
    h.set_options(prec, 1e-12, 1e-12, 1)
    sdg.lib().sdg_pressure_cg(h.h, x, y, None, None)
    print(sdg.lib().sdg_last_error().decode())
"""

GPU = """
import numpy as np, torch
from oracle import Grid, Oracle
from paper_1602_05806_gb300 import sdg
L = (6.0, 5.0, 7.0)[:{dim}]
o = Oracle(Grid({dim}, {n}, L), {N}, 0.05, 0.6, 1e-3)
h = sdg.Handle({dim}, {n}, L, {N}, 0.05, 0.6, 1e-3)
rng = np.random.default_rng(1)
b = o.viscous_apply(rng.standard_normal(o.shape))
x0 = rng.standard_normal(o.shape)
dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
for prec in (0, 1):
    h.set_options(prec, 1e-12, 1e-12, 100000)
    before = h.counters()["launches"]
    X = dev(x0)
    info = h.viscous_cg(dev(b), X)
    launches = h.counters()["launches"] - before
    res = np.linalg.norm(b - o.viscous_apply(X.cpu().numpy())) / np.linalg.norm(b)
    bound = max(1e-12, 10.0 * max(info["floor_res"], info["eval_res"]))
    assert info["status"] == 0 and res <= 1.01 * bound + 1e-13, (res, info)
    assert launches >= 2 * info["iters"] > 0, (launches, info)
print("ok")
"""


@pytest.mark.parametrize("n,N", GRIDS)
def test_refused(tmp_path, n, N):
    build.build()
    out = fake_runtime.run(CPU.format(dim=len(n), n=n, N=N), str(tmp_path), SDG_FAKE_DEVICE="1", SDG_REFUSE_COOPERATIVE="1")
    assert out[:2] == ["CG host loop ran past maxit without a device stop"] * 2


@pytest.mark.gpu
@pytest.mark.parametrize("n,N", GRIDS)
def test_refused_solves(tmp_path, n, N):
    out = fake_runtime.run(GPU.format(dim=len(n), n=n, N=N), str(tmp_path), SDG_REFUSE_COOPERATIVE="1")
    assert out[0] == "ok"
