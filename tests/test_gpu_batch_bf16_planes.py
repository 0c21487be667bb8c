"""Batched BF16 Tikhonov on compressed planes for media that are looked at from some millimetres down, where a few
planes hold most of a measurement: the rounding of the two-term split does not average out there (2e-4 from the exact
solution).  With three terms what is left is FP32 rounding (6e-8), which the solve amplifies by up to
1 / lambda_rel = 1e3.  64 depths: the plan with 16-plane chunks."""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, medium, oracle_grid, rel_l2
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,nt,first", [(16, 3, 256, 12.0), (16, 8, 256, 8.0), (12, 33, 208, 4.0), (8, 64, 256, 2.0)])
def test_deep_media(n, nz, nt, first):
    kw = dict(n=n, nz=nz, nt=nt, dx=0.5, dz=0.5, z_first=first, dt=25.0)
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(grid_kw=kw)), g)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.5, 0.5, first, 25.0))
    try:
        assert 2 * k.planes() <= nt
        rng = np.random.default_rng(nz)
        mu = rng.uniform(0.0, 0.02, (3, nz, n, n)) * (rng.uniform(size=(3, nz, n, n)) < 0.2)
        ms = np.stack([op.forward_fft(wh, v, g) for v in mu])
        want = [so.tikhonov(wh, m, g)[0] for m in ms]
        md = torch.tensor(ms, dtype=torch.float32, device="cuda")
        for steps in (0, 1, 2):
            got = k.reconstruct_batch_tikhonov(md, precision=ctof.BF16, refine=steps)[0].cpu().numpy()
            for a, b in zip(got, want):
                assert rel_l2(a, b) <= 6e-8 * 1e3
    finally:
        k.close()
