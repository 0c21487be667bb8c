"""Time-compressed operator on absorbers below 20 mm, whose response rises by many decades over the early bins: every
bin's plane against the FP64 oracle relative to itself (or to the bin that shares its complex transform: bins 2 i and
2 i + 1 are the two parts of one, on the bins as on the planes), and every depth of the adjoint of early bins relative
to itself.  The products of a window may cancel (csrc/time_fit.h), by 20 at most and by a few as a rule: ten times the
rounding of Q, V and the transforms (6e-8, 6e-8 and 1e-7).  A 32 x 32 scan, from which single calls use the planes;
the oracle takes the handle's own FP64 kernel table (which has its parity tests)."""

import numpy as np
import pytest

from gpu_common import CFG1_OPTICS, oracle_grid
from oracle import operators as op
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 10 * (6e-8 + 6e-8 + 1e-7)


@pytest.mark.parametrize("nz,nt,first", [(48, 256, 40), (64, 256, 56)])
def test_own_scale(nz, nt, first):
    n = 32
    kw = dict(n=n, nz=nz, nt=nt, dx=0.5, dz=0.5, z_first=0.5, dt=25.0)
    g = oracle_grid(kw)
    k = ctof.Kernel(ctof.make_optics(**CFG1_OPTICS), ctof.make_grid(n, nz, nt, 0.5, 0.5, 0.5, 25.0), keep_w=True)
    try:
        wh = op.kernel_spectrum(op._mirror(k.get_w(), n), g)
        assert 2 * k.planes() <= nt
        mu = np.zeros((nz, n, n))
        mu[first:, 4:12, 5:21] = 0.01
        want = op.forward_fft(wh, mu, g)
        got = k.forward(torch.tensor(mu, dtype=torch.float32, device="cuda")).cpu().numpy()
        norms = np.linalg.norm(want, axis=(1, 2)).reshape(-1, 2).max(axis=1).repeat(2)
        seen = norms > 1e-30 * norms.max()
        assert (np.linalg.norm(got - want, axis=(1, 2))[seen] / norms[seen]).max() <= TOL
        m = np.zeros((nt, n, n))
        m[16:20, 3:19, 6:23] = 1.0
        want = op.adjoint_fft(wh, m, g)
        got = k.adjoint(torch.tensor(m, dtype=torch.float32, device="cuda")).cpu().numpy()
        norms = np.linalg.norm(want, axis=(1, 2))
        assert (np.linalg.norm(got - want, axis=(1, 2)) / norms).max() <= TOL
    finally:
        k.close()
