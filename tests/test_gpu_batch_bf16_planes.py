"""Batched BF16 Tikhonov on compressed planes for media that are looked at from some millimetres down, where a few
planes hold most of a measurement.  The yardstick is the two-term split over the time bins (products hi hi, hi lo,
lo hi), done here on the oracle's spectra: the planes may be no further from the exact solution than that, with a
quarter for the scatter of rounding errors and 2e-5 for the FP32 rounding of the rest (twice the FP32 path's 1e-5).
64 depths: the plan with 16-plane chunks."""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, medium, oracle_grid, rel_l2
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def split(a):
    f = torch.tensor(np.ascontiguousarray(a), dtype=torch.float32)
    hi = f.bfloat16().float()
    return hi.double().numpy(), (f - hi).bfloat16().double().numpy()


def two_terms_on_the_bins(wh, m, g, lam):
    w = wh.real
    mh = np.fft.fft2(op._pad(m, g), axes=(-2, -1))
    (w0, w1), (r0, r1), (i0, i1) = split(w), split(mh.real), split(mh.imag)
    dot = lambda a, b: np.einsum("tzyx,tyx->yxz", a, b)
    b = sum(dot(x, r) + 1j * dot(x, i) for x, r, i in ((w0, r0, i0), (w0, r1, i1), (w1, r0, i0)))
    x = np.linalg.solve(so.gram(w) + lam * np.eye(g.nz), b[..., None])[..., 0]
    return np.fft.ifft2(np.moveaxis(x, -1, 0), axes=(-2, -1)).real[:, :g.n, :g.n]


@pytest.mark.parametrize("n,nz,nt,first", [(16, 3, 256, 12.0), (16, 8, 256, 8.0), (16, 3, 368, 0.5), (8, 64, 256, 2.0)])
def test_no_further_off_than_on_the_bins(n, nz, nt, first):
    kw = dict(n=n, nz=nz, nt=nt, dx=0.5, dz=0.5, z_first=first, dt=25.0)
    g = oracle_grid(kw)
    wh = op.kernel_spectrum(op.kernel_offsets(g, medium(grid_kw=kw)), g)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.5, 0.5, first, 25.0))
    try:
        assert 2 * k.planes() <= nt
        rng = np.random.default_rng(nz)
        mu = rng.uniform(0.0, 0.02, (4, nz, n, n)) * (rng.uniform(size=(4, nz, n, n)) < 0.2)
        ms = np.stack([op.forward_fft(wh, v, g) for v in mu])
        exact, lam = zip(*[so.tikhonov(wh, m, g)[:2] for m in ms])
        exact = np.stack(exact)
        bins = rel_l2(np.stack([two_terms_on_the_bins(wh, m, g, lam[0]) for m in ms]), exact)
        md = torch.tensor(ms, dtype=torch.float32, device="cuda")
        for steps in (1, 2):
            got = k.reconstruct_batch_tikhonov(md, precision=ctof.BF16, refine=steps)[0].cpu().numpy()
            assert rel_l2(got, exact) <= 1.25 * bins + 2e-5, (steps, bins)
    finally:
        k.close()
