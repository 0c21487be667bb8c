"""What the Tikhonov solves keep on a handle is kept once, whichever operator (bins or planes) a call runs on."""

import ctypes

import pytest

from gpu_common import CFG1_OPTICS
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_precisions_share_workspace_and_tables():
    n, nz, nt, batch = 32, 16, 256, 32
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.5, 0.5, 0.5, 25.0))
    try:
        assert 2 * k.planes() <= nt
        m = torch.rand((batch, nt, n, n), device="cuda")
        out = torch.empty((batch, nz, n, n), device="cuda")
        solve = lambda precision: k.reconstruct_batch_tikhonov(m, precision=precision, out=out)
        solve(ctof.FP8E4M3)
        want = out.clone()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        solve(ctof.BF16)
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] < 1 << 20
        solve(ctof.FP8E4M3)
        assert torch.equal(out, want)
    finally:
        k.close()


def test_device_bytes_follow_what_is_made_on_first_use():
    n, nz, nt, batch = 32, 16, 256, 64
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.5, 0.5, 0.5, 25.0))
    try:
        def held():
            info = ctof.KernelInfo()
            assert k._lib.ctof_kernel_get_info(k._h, ctypes.byref(info)) == ctof.OK
            return info.device_bytes

        m = torch.rand((batch, nt, n, n), device="cuda")
        out = torch.empty((batch, nz, n, n), device="cuda")
        torch.cuda.synchronize()
        free, before = torch.cuda.mem_get_info()[0], held()
        k.reconstruct_batch_tikhonov(m, precision=ctof.FP8E4M3, out=out)
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
        # the driver hands memory out in 2 MiB pieces, two allocations
        assert taken - (4 << 20) <= held() - before <= taken
    finally:
        k.close()
