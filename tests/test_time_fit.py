"""Host fit of the time basis (csrc/time_fit.h): compiled here with the C++ compiler and run on synthetic tables."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import operators as op
from oracle import physics as ph

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_11680_gb300", "csrc")
COLUMNS = 16  # row pitch of the device table

SOURCE = r"""
#include "time_fit.h"
extern "C" int fit_table(const double* w, int nt, int nz, int ns, double* q, int* win, int* rank) {
  time_fit::Basis b;
  if (!time_fit::fit(std::vector<double>(w, w + (size_t)nt * nz * ns), nt, nz, ns, &b)) return -1;
  std::copy(b.q.begin(), b.q.end(), q);
  for (size_t i = 0; i < b.win.size(); ++i) {
    const int row[4] = {b.win[i].begin, b.win[i].end, b.win[i].plane, b.win[i].planes};
    std::copy(row, row + 4, win + 4 * i);
  }
  *rank = b.rank;
  return (int)b.win.size();
}
"""


@pytest.fixture(scope="module")
def fit(tmp_path_factory):
    d = tmp_path_factory.mktemp("fit")
    (d / "fit.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "fit.so"),
                    str(d / "fit.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "fit.so"))

    def run(w):
        """w [nt][samples][depths], sample 0 the DC class -> windows (begin, end, plane, planes), Q [nt][16], rank."""
        nt, ns, nz = w.shape
        w = np.ascontiguousarray(w, dtype=np.float64)
        q, win, rank = np.zeros((nt, COLUMNS)), np.zeros((nt, 4), dtype=np.int32), ctypes.c_int()
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        n = lib.fit_table(ptr(w), nt, nz, ns, ptr(q), ptr(win), ctypes.byref(rank))
        assert n > 0
        return win[:n], q, rank.value

    return run


def project(w, win, q):
    out = np.zeros_like(w)
    for a, b, _, r in win:
        out[a:b] = np.einsum("tj,uj,usz->tsz", q[a:b, :r], q[a:b, :r], w[a:b])
    return out


@pytest.mark.parametrize("nt", [49, 60])
def test_seventeen_bins_of_rank_sixteen(fit, nt):
    """A window one bin longer than the table has columns, one rank short of its bins: the last one (49 bins), or one
    with bins behind it (60: the response falls at bin 49)."""
    rng = np.random.default_rng(nt)
    w = rng.uniform(0.5, 1.0, (nt, 8, 4))
    w[48] = np.tensordot(rng.uniform(0.0, 0.1, 16), w[32:48], axes=(0, 0))
    w[49:] *= 1e-5
    win, q, rank = fit(w)
    assert [32, 49] in win[:, :2].tolist()
    assert win[:, 3].max() <= COLUMNS and rank == win[:, 3].sum()
    assert np.abs(project(w, win, q) - w).max() <= 1e-9


@pytest.mark.parametrize("nz,nt,d,dt", [(48, 256, 0.5, 25.0), (64, 512, 0.5, 25.0), (40, 160, 1.0, 50.0)])
def test_every_bin_and_depth_in_fp32(fit, nz, nt, d, dt):
    """The stored FP32 factors give every bin of every depth's DC response back, also where a deep layer's response
    rises by many decades within a window.  The products may cancel, by 20 at most and by a few as a rule: ten times the
    rounding of Q, V and their sum (6e-8 each)."""
    g = op.Grid(8, nz, nt, d, d, d, dt)
    wh = op.kernel_spectrum(op.kernel_offsets(g, ph.Medium(0.01, 1.0, 1.4, r_min=0.5 * d)), g)
    w = np.ascontiguousarray(np.moveaxis(wh.real.reshape(nt, nz, -1), 2, 1)[:, ::5])
    win, q, rank = fit(w)
    assert win[-1, 1] == nt and rank == win[:, 3].sum()
    assert 2 * rank <= nt
    dc = w[:, 0]
    for a, b, _, r in win:
        qs = q[a:b, :r].astype(np.float32)
        assert np.abs(q[a:b, :r].T @ q[a:b, :r] - np.eye(r)).max() <= 1e-12
        v = (q[a:b, :r].T @ dc[a:b]).astype(np.float32)
        got = np.zeros((b - a, nz), dtype=np.float32)
        for j in range(r):
            got += qs[:, j, None] * v[j]
        seen = dc[a:b] > 1e-30 * dc[a:b].max(axis=1, keepdims=True)
        assert (np.abs(got - dc[a:b]) / dc[a:b])[seen].max() <= 10 * 3 * 6e-8
