"""Class blocks that fit the slots of the one-warp-per-class x-update but not those of the adjoint or the Tikhonov
solve, on handles that keep the bins (absorbing media, whose responses do not compress in time): every call against
the FP64 oracle at the FP32 path's 1e-5.  The Tikhonov solve amplifies the FP32 rounding (6e-8) of its right-hand
side by up to 1 / lambda_rel = 1e3 and sums over nt bins: 6e-5 sqrt(nt / 64)."""

import numpy as np
import pytest

from gpu_common import medium, oracle_grid, rel_l2
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mua,nz,nt,d,dt", [(0.05, 32, 220, 0.5, 50.0), (0.02, 48, 136, 1.0, 50.0),
                                            (0.02, 32, 220, 1.0, 100.0), (0.1, 16, 400, 0.5, 50.0)])
def test_large_blocks_on_the_bins(mua, nz, nt, d, dt):
    n = 16
    kw = dict(n=n, nz=nz, nt=nt, dx=d, dz=d, z_first=d, dt=dt)
    optics = dict(mua=mua, musp=1.0, n=1.4)
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(optics, kw)), g)
    k = ctof.Kernel(ctof.make_optics(**optics), ctof.make_grid(n, nz, nt, d, d, d, dt))
    try:
        assert k.planes() == nt
        rng = np.random.default_rng(nt)
        mu = rng.uniform(0.0, 0.02, (nz, n, n)) * (rng.uniform(size=(nz, n, n)) < 0.3)
        m = op.forward_fft(wh, mu, g)
        md = torch.tensor(m, dtype=torch.float32, device="cuda")
        assert rel_l2(k.forward(torch.tensor(mu, dtype=torch.float32, device="cuda")).cpu().numpy(), m) <= 1e-5
        assert rel_l2(k.adjoint(md).cpu().numpy(), op.adjoint_fft(wh, m, g)) <= 1e-5
        got = k.reconstruct(md, ctof.tikhonov_params()).cpu().numpy()
        assert rel_l2(got, so.tikhonov(wh, m, g)[0]) <= 6e-5 * np.sqrt(nt / 64)
        assert rel_l2(k.reconstruct(md, ctof.admm_params(6)).cpu().numpy(), so.admm(wh, m, g, 6)[0]) <= 1e-5
        got = k.reconstruct(md, ctof.fista_params(6)).cpu().numpy()
        assert rel_l2(got, so.fista_l1(wh, m, g, 6)[0]) <= 1e-5
    finally:
        k.close()


@pytest.mark.parametrize("nz,nt,name", [(6, 32, "k_contract_warp"), (64, 100, "k_contract_admm_pipe")])
def test_name_of_the_x_update(nz, nt, name):
    k = ctof.Kernel(ctof.make_optics(), ctof.make_grid(8, nz, nt, 1.0, 1.0, 1.0, 50.0))
    try:
        assert k.planes() == nt and k.admm_kernel() == name
    finally:
        k.close()
