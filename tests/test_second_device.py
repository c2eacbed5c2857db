"""Handles on two devices of one process: kernels whose shared memory has to be
allowed per device launch on the second one too.  CPU: the runtime is a
stand-in that refuses a launch beyond 48 KB where that was not allowed on the
current device (tests/fake_cudart.c); its kernels do nothing, so a solve with
cooperative launches ends at its one residual replacement, and one with
launches per iteration at the host's own cap on batches."""
import pytest

from paper_1602_05806_gb300 import build
from tests import fake_runtime

CODE = """
import ctypes, os
from paper_1602_05806_gb300 import sdg
L, rt = sdg.lib(), ctypes.CDLL(os.environ["FAKE"])
for device in (0, 1):
    rt.cudaSetDevice(device)
    h = sdg.Handle({dim}, {n}, (1.0,) * 3, {N}, 0.1, 0.6, 0.01)
    x, y = (ctypes.create_string_buffer(8 * h.ndof) for _ in range(2))
    for fp32 in (0, 1):
        print(device, "apply", L.sdg_pressure_apply(h.h, x, y, fp32, None), L.sdg_last_error().decode())
    h.set_mixed_options(0.5, 1)
    for prec in (0, 1):
        for form in (1, 2):
            h.set_options(prec, 1e-12, 1e-12, 1)
            h.set_iteration_form(form)
            rc = L.sdg_pressure_cg(h.h, x, y, None, None)
            print(device, "cg", prec, form, rc, L.sdg_last_error().decode() if rc else "")
"""


# k_apply and its spread CG operator (2D FP64), k_apply3m, k_cg_res and
# k_cg_resid above 48 KB (13^3 cells at N = 3), k_cg_big
@pytest.mark.parametrize("n,N", [((64, 64), 5), ((60, 50), 7), ((100, 90), 6), ((128, 128), 7), ((13, 12, 11), 3), ((24, 24, 24), 4),
                                 ((12, 12, 12), 5)])
def test_second_device(tmp_path, n, N):
    build.build()
    out = fake_runtime.run(CODE.format(dim=len(n), n=n, N=N), str(tmp_path), SDG_FAKE_DEVICE="1")
    seen = {d: [line[2:] for line in out if line.startswith(d)] for d in ("0", "1")}
    assert len(seen["0"]) == 6
    for line in seen["0"] + seen["1"]:
        assert "CUDA error" not in line, line
