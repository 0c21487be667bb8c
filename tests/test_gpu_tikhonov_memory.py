"""What the Tikhonov solves keep on a handle is kept once, whichever operator (bins or planes) a call runs on."""

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
