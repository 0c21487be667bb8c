"""ADMM and the learned solver's operator on a circular (periodic) scan, whose
N columns fill the whole P-wide FFT row (a linear scan fills at most half of
it), against the FP64 oracle: 1e-5 as in test_gpu_parity.py; the learned
output against the oracle that rounds to BF16 where the device stores, 2e-4 as
in test_gpu_learned.py."""

import numpy as np
import pytest

from gpu_common import device_kernel, oracle_kernel, rel_l2
from oracle import learned as ol
from oracle import operators as op
from oracle import solvers as so
from paper_2101_11680_gb300 import ctof, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _measurement(seed):
    g, _, wh = oracle_kernel("circ")
    rng = np.random.default_rng(seed)
    mu = rng.uniform(0.0, 0.02, (g.nz, g.n, g.n)) * (rng.uniform(size=(g.nz, g.n, g.n)) < 0.2)
    return g, wh, op.forward_fft(wh, mu, g)


def test_circular_admm():
    g, wh, m = _measurement(21)
    got = device_kernel("circ").reconstruct(torch.tensor(m, dtype=torch.float32, device="cuda"), ctof.admm_params(40))
    assert rel_l2(got.cpu().numpy(), so.admm(wh, m, g, 40)[0]) <= 1e-5


def test_circular_learned():
    g, wh, m = _measurement(22)
    s = so.spectral_norm(wh)
    theta = ol.bf16(synth.learned_init(2, seed=3))
    net = ctof.Learned(2, theta)
    got = net.reconstruct(device_kernel("circ"), torch.tensor(m[None], dtype=torch.float32, device="cuda"))
    want = ol.unrolled(theta, 2, lambda x: op.forward_fft(wh / s, x, g), lambda r: op.adjoint_fft(wh / s, r, g), m / s,
                       rnd=ol.bf16)
    assert rel_l2(got[0].cpu().numpy(), want) <= 2e-4
