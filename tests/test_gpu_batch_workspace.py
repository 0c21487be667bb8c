"""Batched Tikhonov with volumes x bins (and volumes x depths) off the row passes' plane pitch of 16, on grids
whose handles keep the bins: every volume against the single-volume solve at the precision form's stated 1e-3."""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, rel_l2
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [ctof.BF16, ctof.FP8E4M3])
@pytest.mark.parametrize("n,nz,nt,batch", [(20, 6, 23, 5), (12, 9, 7, 17), (44, 5, 30, 3)])
def test_ragged_planes(n, nz, nt, batch, prec):
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 1.0, 1.0, 1.0, 50.0))
    try:
        rng = np.random.default_rng(nt)
        mu = torch.tensor(rng.uniform(0.0, 0.02, (batch, nz, n, n)), dtype=torch.float32, device="cuda")
        m = torch.stack([k.forward(v) for v in mu])
        got = k.reconstruct_batch_tikhonov(m, precision=prec)[0].cpu().numpy()
        for b in range(batch):
            want = k.reconstruct(m[b], ctof.tikhonov_params()).cpu().numpy()
            assert rel_l2(got[b], want) <= 1e-3
    finally:
        k.close()
