"""The time-compressed operator (W_hat = Q V) against the FP64 oracle, bin by
bin and depth by depth: the factorisation must not trade the accuracy of weak
bins or deep layers for that of the strong ones.

Tolerance: the FP32 path's stated 1e-5, here for every bin's plane and every
depth's layer on its own.  A bin's error is relative to the largest plane from
it to twice its index (a window of the basis spans at most that, and on the
rising edge of a deep absorber's response FP32 keeps no more).  Grids: even and
odd scan sizes (paired and single scan points per lane), bins that do not fill
the last window, a scan whose planes are half its bins, circular convolution."""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, medium, oracle_grid, rel_l2
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = {
    "even": dict(n=40, nz=6, nt=208, dx=0.5, dz=0.9, z_first=0.5, dt=25.0),
    "odd": dict(n=41, nz=5, nt=211, dx=0.5, dz=1.1, z_first=0.5, dt=25.0),
    "half": dict(n=66, nz=4, nt=96, dx=0.5, dz=1.5, z_first=0.5, dt=25.0),
    "circular": dict(n=128, nz=3, nt=200, dx=0.5, dz=2.0, z_first=0.5, dt=25.0, mode="circular"),
}


@pytest.fixture(scope="module", params=list(GRIDS))
def problem(request):
    from paper_2101_11680_gb300 import build as B
    B.build()
    kw = GRIDS[request.param]
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(grid_kw=kw), nodes=8, sub=4), g)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS),
                    ctof.make_grid(kw["n"], kw["nz"], kw["nt"], kw["dx"], kw["dz"], kw["z_first"], kw["dt"],
                                   mode=kw.get("mode", "linear")))
    yield g, wh, k
    k.close()


def test_forward_bin_by_bin(problem):
    g, wh, k = problem
    rng = np.random.default_rng(3)
    for z in (0, g.nz - 1):
        mu = np.zeros((g.nz, g.n, g.n))
        mu[z] = rng.uniform(0.0, 0.02, (g.n, g.n)) * (rng.uniform(size=(g.n, g.n)) < 0.3)
        got = k.forward(torch.tensor(mu, dtype=torch.float32, device="cuda")).cpu().numpy()
        want = op.forward_fft(wh, mu, g)
        norms = np.linalg.norm(want, axis=(1, 2))
        for t in range(g.nt):
            err = np.linalg.norm(got[t] - want[t])
            assert err <= 1e-5 * norms[t:2 * t + 16].max(), (z, t)


def test_adjoint_depth_by_depth_for_gated_bins(problem):
    g, wh, k = problem
    rng = np.random.default_rng(4)
    shape = np.abs(wh[:, :, 0, 0]).max(axis=1)  # the response's own fall over the bins
    for a, b in ((0, g.nt), (g.nt // 4, g.nt // 2), (3 * g.nt // 4, g.nt)):
        m = np.zeros((g.nt, g.n, g.n))
        m[a:b] = rng.uniform(0.5, 1.0, (b - a, g.n, g.n)) * shape[a:b, None, None]
        # a measurement that starts 4 bytes off an 8-byte boundary, as a slice of a larger record may
        rec = torch.zeros(m.size + 1, device="cuda")
        rec[1:] = torch.tensor(m, dtype=torch.float32).reshape(-1)
        got = k.adjoint(rec[1:].reshape(m.shape)).cpu().numpy()
        want = op.adjoint_fft(wh, m, g)
        for z in range(g.nz):
            assert rel_l2(got[z], want[z]) <= 1e-5, (a, z)


def test_solvers(problem):
    g, wh, k = problem
    rng = np.random.default_rng(5)
    mu = rng.uniform(0.0, 0.02, (g.nz, g.n, g.n)) * (rng.uniform(size=(g.nz, g.n, g.n)) < 0.1)
    m = op.forward_fft(wh, mu, g)
    md = torch.tensor(m, dtype=torch.float32, device="cuda")
    scale = max(1.0, np.sqrt(g.nt / 64))  # FP32 sums of W^T m over nt bins
    assert rel_l2(k.reconstruct(md, ctof.tikhonov_params()).cpu().numpy(), so.tikhonov(wh, m, g)[0]) <= 1e-5 * scale
    assert rel_l2(k.reconstruct(md, ctof.admm_params(8)).cpu().numpy(), so.admm(wh, m, g, 8)[0]) <= 1e-5
    assert rel_l2(k.reconstruct(md, ctof.fista_params(10)).cpu().numpy(), so.fista_l1(wh, m, g, 10)[0]) <= 1e-5


@pytest.mark.parametrize("volumes", [1, 64])
def test_projection_groups(problem, volumes):
    """Batched Tikhonov with few and with many projection CTAs, at the precision form's stated 1e-3."""
    g, wh, k = problem
    rng = np.random.default_rng(6)
    mu = rng.uniform(0.0, 0.02, (2, g.nz, g.n, g.n)) * (rng.uniform(size=(2, g.nz, g.n, g.n)) < 0.1)
    ms = np.stack([op.forward_fft(wh, x, g) for x in mu])
    md = torch.tensor(ms, dtype=torch.float32, device="cuda")
    got = k.reconstruct_batch_tikhonov(md[[0] * (volumes - 1) + [1]].contiguous(), precision=ctof.BF16)[0]
    want = [so.tikhonov(wh, m, g)[0] for m in ms]
    assert rel_l2(got[-1].cpu().numpy(), want[1]) <= 1e-3
    for b in range(0, volumes - 1, 9):
        assert rel_l2(got[b].cpu().numpy(), want[0]) <= 1e-3
