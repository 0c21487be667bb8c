"""Single-volume contractions and x-update, one warp or pair of warps per
frequency class: depths around the 8-row blocks and 4-wide chunks (odd block
counts, one depth, the most), bins around the row sets of the adjoint pass, and
a grid whose classes go several times around the shared-memory ring, against
the FP64 oracle at the FP32 path's 1e-5.  (The Tikhonov solve has its tests at
well-conditioned grids: at these fine depths FP32 rounding of its right-hand
side alone gives up to 3e-5.)"""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, medium, oracle_grid, rel_l2
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,nt", [(8, 1, 40), (8, 17, 33), (9, 24, 40), (8, 33, 63), (8, 40, 48), (9, 49, 31),
                                     (8, 55, 40), (8, 64, 48), (72, 9, 23)])
def test_sizes(n, nz, nt):
    from paper_2101_11680_gb300 import build as B
    B.build()
    kw = dict(n=n, nz=nz, nt=nt, dx=0.6, dz=0.4, z_first=0.4, dt=30.0)
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(grid_kw=kw)), g)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.6, 0.4, 0.4, 30.0))
    try:
        rng = np.random.default_rng(nz)
        mu = rng.uniform(0.0, 0.02, (nz, n, n)) * (rng.uniform(size=(nz, n, n)) < 0.3)
        m = op.forward_fft(wh, mu, g)
        dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
        assert rel_l2(k.forward(dev(mu)).cpu().numpy(), m) <= 1e-5
        assert rel_l2(k.adjoint(dev(m)).cpu().numpy(), op.adjoint_fft(wh, m, g)) <= 1e-5
        got = k.reconstruct(dev(m), ctof.admm_params(6)).cpu().numpy()
        assert rel_l2(got, so.admm(wh, m, g, 6)[0]) <= 1e-5
    finally:
        k.close()


def test_waits_give_up_and_recover():
    """With no polls allowed the kernels stop, drain and report; with the default limit the call is right again."""
    kw = dict(n=16, nz=6, nt=32, dx=1.0, dz=1.0, z_first=1.0, dt=50.0)
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(grid_kw=kw)), g)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(16, 6, 32, 1.0, 1.0, 1.0, 50.0))
    try:
        m = np.random.default_rng(1).uniform(0.0, 1.0, (32, 16, 16))
        md = torch.tensor(m, dtype=torch.float32, device="cuda")
        k.set_wait_limit(0)
        k.adjoint(md)
        with pytest.raises(ctof.CtofError) as e:
            k.sync_status()
        assert e.value.status == ctof.ETIMEOUT
        k.set_wait_limit(1 << 24)
        got = k.adjoint(md)
        k.sync_status()
        assert rel_l2(got.cpu().numpy(), op.adjoint_fft(wh, m, g)) <= 1e-5
    finally:
        k.close()
