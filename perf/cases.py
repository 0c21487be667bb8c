"""The work this library does for its users, as cases that can be timed and checked.

A case is one pass through the public entry points of ``paper_2101_11680_gb300.ctof``: an operator application, a
reconstruction, a batch of either, or a training gradient.  Geometries follow the repository's own configurations
(config 1: 32 x 32 x 16 voxels, 64 bins of 50 ps at 1 mm; config 2: 128 x 128 x 48 voxels, 256 bins of 25 ps at 0.5 mm;
the 64-depth x 512-bin class block of the precision form; the 64 x 64 scan the learned form is trained on).  Inputs are
synthetic: ellipsoid phantoms and photon-counted diffuse time curves.

``exact`` restates the model in 64 bits with plain torch: the kernel table from the closed-form diffusion Green's
functions, its spectrum, and each solver step by step.
"""

import math
import os
import random

import numpy as np
import torch

from paper_2101_11680_gb300 import ctof

OPTICS = {"mua": 0.01, "musp": 1.0, "n": 1.4}
MU0 = 0.01          # network input scale of the learned solver [1/mm]
CHANNELS = ((1, 16), (16, 16), (16, 16), (16, 1))
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(ctof.__file__)), "weights", "learned_s10.npz")


# ---- the cases ----

def _grid(n, nz, nt, pitch=0.5, dt=25.0, mode="linear"):
    return {"n": n, "nz": nz, "nt": nt, "pitch": pitch, "dt": dt, "mode": mode}


def listed():
    return [
        # one forward projection of a small scan (config 1), as an interactive simulator issues them: latency
        {"name": "forward_scan32", "path": "forward", **_grid(32, 16, 64, 1.0, 50.0)},
        # forward projection on the largest linear FFT grid (256 x 256 scan, P = 512)
        {"name": "forward_scan256", "path": "forward", **_grid(256, 32, 128)},
        # back projection at the headline geometry (config 2)
        {"name": "adjoint_scan128", "path": "adjoint", **_grid(128, 48, 256)},
        # quick-look reconstruction of one odd-sized scan: neither power-of-two rows nor whole plane tiles
        {"name": "tikhonov_scan100", "path": "tikhonov", **_grid(100, 37, 203)},
        # the headline reconstruction: 100 ADMM iterations with TV at config 2
        {"name": "admm_scan128", "path": "admm", **_grid(128, 48, 256), "iters": 100},
        # independent problems of uneven sizes and optics in one call (the batching form's mix, up to 128 x 128)
        {"name": "admm_mixed6", "path": "admm_mixed", "count": 6, "problems": 11, "iters": 50},
        # the paper's own solver on its source-multiplexed measurement, 64 x 64 scan
        {"name": "fista_mux64", "path": "fista", **_grid(64, 32, 128), "iters": 100, "multiplexed": True},
        # spectra-level A and A^T for sixteen volumes that share a kernel, as iterative solvers on spectra use them
        {"name": "contract_batch16", "path": "contract", **_grid(128, 48, 256), "batch": 16},
        # precision form, BF16 contraction with two refinement steps, at its own class block
        {"name": "tikhonov_bf16_batch16", "path": "tikhonov_batch", **_grid(128, 64, 512), "batch": 16,
         "precision": "bf16"},
        # precision form, FP8, a ragged batch (one full chunk of sixteen volumes and a part)
        {"name": "tikhonov_fp8_batch21", "path": "tikhonov_batch", **_grid(64, 32, 256), "batch": 21,
         "precision": "fp8"},
        # learned form, inference: two stages of the trained solver on sixteen config-2 volumes
        {"name": "learned_stages2", "path": "learned", **_grid(128, 48, 256), "batch": 16, "stages": 2},
        # learned form, training: loss and gradients of a batch of four at the training geometry
        {"name": "learned_grad4", "path": "learned_grad", **_grid(64, 48, 256), "batch": 4, "stages": 2},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    path = rng.choice(["forward", "forward", "adjoint", "adjoint", "tikhonov", "tikhonov", "admm", "admm", "admm_mixed",
                       "fista", "contract", "contract", "tikhonov_batch", "tikhonov_batch", "learned", "learned_grad"])
    if path == "admm_mixed":
        return {"path": path, "count": rng.randint(2, 6), "problems": rng.randint(100, 10 ** 6),
                "iters": rng.randint(10, 50)}
    pitch, dt = rng.choice([(0.5, 25.0), (0.7, 33.0), (1.0, 50.0)])
    mode = "linear"
    n = _log_int(rng, 8, 128)
    if path in ("forward", "adjoint", "tikhonov"):
        n = _log_int(rng, 8, 256)
        if rng.random() < 0.25:
            mode, n = "circular", rng.choice([32, 64, 128, 256])
    elif path.startswith("learned"):
        n = 16 * rng.randint(1, 8 if path == "learned" else 4)
    nz = _log_int(rng, 2, 64)
    nt = _log_int(rng, 8, 512)
    # no larger table than config 2's
    while n * n * nz * nt > 128 * 128 * 48 * 256:
        if nt >= 4 * nz:
            nt = nt * 3 // 4
        else:
            nz = max(1, nz * 3 // 4)
    case = {"path": path, **_grid(n, nz, nt, pitch, dt, mode)}
    if path == "admm":
        case["iters"] = rng.randint(10, 100)
    elif path == "fista":
        mux = rng.random() < 0.5
        if mux:
            case["n"] = n = max(8, n // 8 * 8)
        case.update(iters=rng.randint(5, 40), multiplexed=mux)
    elif path == "contract":
        case["batch"] = rng.randint(1, 20)
    elif path == "tikhonov_batch":
        case.update(batch=rng.randint(1, 24), precision=rng.choice(["bf16", "fp8", "fp32"]))
    elif path == "learned":
        case.update(batch=rng.randint(1, 16), stages=2)
    elif path == "learned_grad":
        case.update(batch=rng.randint(1, 4), stages=2)
    return case


def _problems(case):
    """The uneven problems of a mixed batch: grids and optics as the batching form draws them."""
    rng = random.Random(case["problems"])
    out = []
    for _ in range(case["count"]):
        n = rng.choice([32, 48, 64, 96, 128])
        out.append({**_grid(n, rng.randint(8, 40), rng.randint(48, 200)), "mua": rng.uniform(0.005, 0.02),
                    "musp": rng.uniform(0.5, 2.0)})
    return out


# ---- inputs ----

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(gen, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)


def _volume(case, gen):
    """One to eight smooth-edged absorbing ellipsoids of 0.005 .. 0.02 / mm (float32 [nz][n][n])."""
    n, nz, d = case["n"], case["nz"], case["pitch"]
    x = torch.arange(n, device="cuda", dtype=torch.float32) * d
    z = (torch.arange(nz, device="cuda", dtype=torch.float32) + 1) * d
    p = _uniform(gen, (8, 8), 0.0, 1.0).cpu().tolist()
    vol = torch.zeros((nz, n, n), device="cuda")
    for q in p[:1 + int(8 * p[0][7]) % 8]:
        ext, dep = (n - 1) * d, nz * d
        r = ((x[None, None, :] - q[0] * ext) / (1 + 3 * q[1])) ** 2
        r = r + ((x[None, :, None] - q[2] * ext) / (1 + 3 * q[3])) ** 2
        r = r + ((z[:, None, None] - q[4] * dep) / (1 + 3 * q[5])) ** 2
        vol = torch.maximum(vol, (0.005 + 0.015 * q[6]) * torch.clamp(4.0 * (1.0 - r), 0.0, 1.0))
    return vol


def _measurement(case, gen):
    """Differential time curves of a few absorbers, counted as photons (Poisson, peak 1e5 counts; peak 5e-4 in the units of A mu).

    Each absorber at depth z darkens the scan with the diffuse shape t^-5/2 exp(-(rho^2 + z^2) / 2 D c t - mua c t)."""
    n, nt, d, dt = case["n"], case["nt"], case["pitch"], case["dt"]
    c, dc = 0.299792458 / 1.4, 0.299792458 / 1.4 / (3 * 1.01)
    x = torch.arange(n, device="cuda", dtype=torch.float32) * d
    t = (torch.arange(nt, device="cuda", dtype=torch.float32) + 0.5) * dt
    p = _uniform(gen, (4, 4), 0.0, 1.0).cpu().tolist()
    m = torch.zeros((nt, n, n), device="cuda")
    for q in p:
        rho2 = (x[None, :] - q[0] * (n - 1) * d) ** 2 + (x[:, None] - q[1] * (n - 1) * d) ** 2
        z2 = (1.0 + 6.0 * q[2]) ** 2
        tt = t[:, None, None]
        m += (0.2 + q[3]) * (z2 + 1) ** 2 * tt ** -2.5 * torch.exp(-(rho2 + z2) / (2 * dc * tt) - 0.01 * c * tt)
    top = float(m.max())
    return torch.poisson(m * (1e5 / top), generator=gen) * (5e-4 / 1e5)


def _stack(make, case, gen, count):
    return torch.stack([make(case, gen) for _ in range(count)]).contiguous()


def _learned_params(stages):
    with np.load(WEIGHTS) as f:
        theta = np.asarray(f["theta"], dtype=np.float32)
    weights = sum(ci * co * 27 + co for ci, co in CHANNELS)
    return np.concatenate([theta[:weights], theta[weights:weights + stages]])


def _spectra(case, gen, count, planes, make, ld):
    """Half-plane spectra [count][P (P/2+1)][ld][2] of zero-padded planes, plane fastest."""
    p = _fft_size(case)
    out = torch.zeros((count, p * (p // 2 + 1), ld, 2), device="cuda")
    for v in range(count):
        f = torch.fft.rfft2(make(case, gen), s=(p, p)).reshape(planes, -1).t()
        out[v, :, :planes] = torch.view_as_real(f.contiguous())
    return out


def _fft_size(case):
    if case["mode"] == "circular":
        return case["n"]
    p = 32
    while p < 2 * case["n"]:
        p *= 2
    return p


def _handle(case):
    grid = ctof.make_grid(case["n"], case["nz"], case["nt"], case["pitch"], case["pitch"], case["pitch"], case["dt"],
                          mode=case["mode"])
    return ctof.Kernel(ctof.make_optics(case.get("mua", OPTICS["mua"]), case.get("musp", OPTICS["musp"]), OPTICS["n"]), grid)


def prepare(case, seed):
    gen, path = _generator(seed), case["path"]
    s = {"case": case, "path": path}
    if path == "admm_mixed":
        probs = _problems(case)
        s["kernels"] = [_handle(p) for p in probs]
        for k in s["kernels"]:
            k.autotune()
        s["m"] = [_measurement(p, gen) for p in probs]
        s["params"] = ctof.admm_params(case["iters"])
        return s
    k = s["kernel"] = _handle(case)
    batch = case.get("batch", 1)
    if path == "forward":
        s["mu"] = _volume(case, gen)
    elif path in ("adjoint", "tikhonov", "admm", "fista"):
        s["m"] = _measurement(case, gen)
    elif path == "contract":
        s["z"] = _spectra(case, gen, batch, case["nz"], _volume, k.ldz)
        s["t"] = _spectra(case, gen, batch, case["nt"], _measurement, k.ldt)
        s["out_t"], s["out_z"] = torch.zeros_like(s["t"]), torch.zeros_like(s["z"])
    else:
        s["m"] = _stack(_measurement, case, gen, batch)
    if path == "tikhonov":
        s["params"] = ctof.tikhonov_params()
    elif path == "admm":
        s["params"] = ctof.admm_params(case["iters"])
        k.autotune()
    elif path == "fista":
        s["params"] = ctof.fista_params(case["iters"], multiplexed=case["multiplexed"])
    elif path.startswith("learned"):
        s["net"] = ctof.Learned(case["stages"], _learned_params(case["stages"]))
        if path == "learned_grad":
            s["mu"] = _stack(_volume, case, gen, batch)
    return s


def run(s):
    path = s["path"]
    if path == "forward":
        return s["kernel"].forward(s["mu"])
    if path == "adjoint":
        return s["kernel"].adjoint(s["m"])
    if path in ("tikhonov", "admm", "fista"):
        return s["kernel"].reconstruct(s["m"], s["params"])
    if path == "admm_mixed":
        return ctof.reconstruct_batch(s["kernels"], s["m"], s["params"])
    if path == "contract":
        return [s["kernel"].contract_forward_batch(s["z"], out=s["out_t"]),
                s["kernel"].contract_adjoint_batch(s["t"], out=s["out_z"])]
    if path == "tikhonov_batch":
        precision = {"bf16": ctof.BF16, "fp8": ctof.FP8E4M3, "fp32": ctof.FP32}[s["case"]["precision"]]
        return s["kernel"].reconstruct_batch_tikhonov(s["m"], precision=precision)[0]
    if path == "learned":
        return s["net"].reconstruct(s["kernel"], s["m"])
    loss, grad = s["net"].loss_grad(s["kernel"], s["m"], s["mu"])
    return {"loss": loss, "grad": grad}


# ---- what a pass cannot do without ----

def _counts(case):
    """Per volume: kernel spectrum bytes (one matrix per frequency class), plane bytes, contraction and FFT operations."""
    n, nz, nt, p = case["n"], case["nz"], case["nt"], _fft_size(case)
    q = p // 2 + 1
    freqs, classes = p * q, q * (q + 1) // 2
    fft = 2.5 * p * p * math.log2(p * p)  # one real 2-D transform
    return {"w": 4.0 * classes * nt * nz, "h": 4.0 * classes * nz * nz, "mu": 4.0 * nz * n * n, "m": 4.0 * nt * n * n,
            "xp": 4.0 * nz * p * p, "freqs": freqs, "mul": 4.0 * freqs * nt * nz, "solve": 4.0 * freqs * nz * nz,
            "fft_z": nz * fft, "fft_t": nt * fft}


def _admm_work(case, iters):
    c = _counts(case)
    # per iteration: the class matrices and m read once; the multipliers u1 (scan), u2 (three gradients), u3 read and written
    per = {"bytes": c["w"] + c["h"] + 3 * c["m"] + 8 * c["xp"],
           "flops": 2 * c["mul"] + c["solve"] + 2 * c["fft_z"] + 2 * c["fft_t"]}
    return {"bytes": iters * per["bytes"] + c["m"] + c["mu"], "flops": iters * per["flops"]}


def work(case):
    path = case["path"]
    if path == "admm_mixed":
        parts = [_admm_work(p, case["iters"]) for p in _problems(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    c, b = _counts(case), case.get("batch", 1)
    one = {"bytes": c["mu"] + c["m"], "flops": c["mul"] + c["fft_z"] + c["fft_t"]}
    if path in ("forward", "adjoint"):
        return {"bytes": c["w"] + one["bytes"], "flops": one["flops"]}
    if path == "tikhonov":
        return {"bytes": c["w"] + c["h"] + one["bytes"], "flops": one["flops"] + c["solve"]}
    if path == "admm":
        return _admm_work(case, case["iters"])
    if path == "fista":
        return {"bytes": case["iters"] * (2 * c["w"] + c["m"] + 4 * c["mu"]), "flops": case["iters"] * 2 * one["flops"]}
    if path == "contract":
        return {"bytes": 2 * c["w"] + 2 * b * 8.0 * c["freqs"] * (case["nz"] + case["nt"]), "flops": 2 * b * c["mul"]}
    if path == "tikhonov_batch":
        return {"bytes": c["w"] + c["h"] + b * one["bytes"], "flops": b * (one["flops"] + 5 * c["solve"])}
    conv = 2.0 * case["n"] ** 2 * case["nz"] * 27 * sum(ci * co for ci, co in CHANNELS)
    s = case["stages"]
    ops = (2 * s - 1) * (1 if path == "learned" else 2)  # x_0 = 0: the first stage needs A^T only
    return {"bytes": ops * c["w"] + b * (one["bytes"] + 2 * s * 16 * c["mu"] / 2 * 3),
            "flops": b * (ops * one["flops"] + s * conv * (1 if path == "learned" else 3))}


# ---- the same results in 64 bits ----

def _table_spectrum(case):
    """W_hat in float64 [P][P/2+1][nt][nz]: the closed-form response integrated over each bin, times the voxel volume."""
    f64 = {"device": "cuda", "dtype": torch.float64}
    n, nz, nt, d, dt, p = case["n"], case["nz"], case["nt"], case["pitch"], case["dt"], _fft_size(case)
    mua, musp, idx = case.get("mua", OPTICS["mua"]), case.get("musp", OPTICS["musp"]), OPTICS["n"]
    c, dif = 0.299792458 / idx, 1.0 / (3.0 * (mua + musp))
    reff = -1.440 / idx ** 2 + 0.710 / idx + 0.668 + 0.0636 * idx
    zb, z0, k, rmin = 2.0 * dif * (1.0 + reff) / (1.0 - reff), 1.0 / (mua + musp), dif * c, 0.5 * d
    offs = p // 2 + 1 if case["mode"] == "circular" else n
    iy, ix = torch.triu_indices(offs, offs, device="cuda")
    rho2 = ((iy.double() * d) ** 2 + (ix.double() * d) ** 2)
    x, w = np.polynomial.legendre.leggauss(8)
    h = dt / 4
    node = torch.tensor(np.concatenate([s * h + 0.5 * h * (x + 1) for s in range(4)]), **f64)
    weight = torch.tensor(np.tile(0.5 * h * w, 4), **f64)
    half = p // 2 + 1
    spec = torch.empty((p, half, nt, nz), **f64)
    place = torch.arange(p, device="cuda")
    place = torch.minimum(place, p - place)  # offset that each periodic index holds
    inside = place < offs
    place = torch.where(inside, place, torch.zeros_like(place))
    for j in range(nz):
        z = (j + 1) * d
        r1 = torch.sqrt(rho2 + (z - z0) ** 2).clamp_min(rmin)
        r2 = torch.sqrt(rho2 + (z + z0 + 2 * zb) ** 2).clamp_min(rmin)
        r3 = torch.sqrt(rho2 + z ** 2).clamp_min(rmin)
        r4 = torch.sqrt(rho2 + (z + 2 * zb) ** 2).clamp_min(rmin)
        quad = torch.zeros((nt, offs, offs), **f64)
        terms = []
        for sg, ri in ((1.0, r1), (-1.0, r2)):
            for zj, rj in ((z, r3), (z + 2 * zb, r4)):
                terms.append((sg * zj / (16 * math.pi ** 2 * dif * ri * rj ** 3), ri + rj, rj))
        step = max(1, (1 << 25) // (rho2.numel() * 32))
        for t0 in range(0, nt, step):
            t1 = min(nt, t0 + step)
            t = (torch.arange(t0, t1, **f64)[:, None] * dt + node).reshape(-1, 1)
            wt = (weight / (2.0 * math.sqrt(math.pi * k))).repeat(t1 - t0)[:, None] * t ** -1.5 * torch.exp(-mua * c * t)
            acc = 0.0
            for f, a, rj in terms:
                e = torch.exp(-a * a / (4 * k * t))
                acc = acc + f * e * (a + rj * (a * a / (2 * k * t) - 1.0))
            val = (acc * wt).reshape(t1 - t0, 32, -1).sum(1) * d ** 3
            quad[t0:t1, iy, ix] = val
            quad[t0:t1, ix, iy] = val
        full = quad[:, place][:, :, place] * (inside[:, None] & inside[None, :])
        spec[..., j] = torch.fft.rfft2(full).real.permute(1, 2, 0)
    return spec.reshape(p * half, nt, nz)


class _Model:
    """The operator, its Gram matrices and the lateral transforms in float64."""

    def __init__(self, case):
        self.case, self.n, self.p = case, case["n"], _fft_size(case)
        self.w = _table_spectrum(case)
        self.gram = torch.bmm(self.w.transpose(1, 2), self.w)

    def scale(self):
        return float(torch.linalg.eigvalsh(self.gram[0])[-1].sqrt())

    def fft(self, planes):  # [k][a][b] -> [freq][k] complex
        return torch.fft.rfft2(planes, s=(self.p, self.p)).reshape(planes.shape[0], -1).t()

    def ifft(self, spec):
        p = self.p
        return torch.fft.irfft2(spec.t().reshape(-1, p, p // 2 + 1), s=(p, p))

    def crop(self, planes):
        return planes[:, :self.n, :self.n]

    @staticmethod
    def mul(mats, spec):  # [freq][a][b] real times [freq][b] complex
        return torch.view_as_complex(torch.bmm(mats, torch.view_as_real(spec.contiguous())).contiguous())

    def forward(self, mu):
        return self.crop(self.ifft(self.mul(self.w, self.fft(mu))))

    def adjoint(self, m):
        return self.crop(self.ifft(self.mul(self.w.transpose(1, 2), self.fft(m))))

    def regularised(self, rel):
        nz = self.gram.shape[-1]
        lam = rel * float(torch.diagonal(self.gram, dim1=1, dim2=2).max())
        return self.gram + lam * torch.eye(nz, device="cuda", dtype=torch.float64)

    def tikhonov(self, m, chol):
        b = self.mul(self.w.transpose(1, 2), self.fft(m))
        x = torch.view_as_complex(torch.cholesky_solve(torch.view_as_real(b.contiguous()), chol).contiguous())
        return self.crop(self.ifft(x))


def _soft(v, thr):
    return torch.sign(v) * (v.abs() - thr).clamp_min(0.0)


def _exact_admm(case, m, iters, rho=1.0):
    f64 = {"device": "cuda", "dtype": torch.float64}
    md, n, p, nz, nt = _Model(case), case["n"], _fft_size(case), case["nz"], case["nt"]
    s = md.scale()
    mn = m.double() / s
    md.w /= s
    beta = 1e-3 * float(md.adjoint(mn).abs().max())
    lap = (2 * torch.sin(math.pi * torch.arange(p, **f64) / p)) ** 2
    diag = (lap[:, None] + lap[None, :p // 2 + 1] + 1.0).reshape(-1)
    dz = torch.zeros((max(nz - 1, 0), nz), **f64)
    i = torch.arange(nz - 1, device="cuda")
    dz[i, i], dz[i, i + 1] = -1.0, 1.0
    hm = md.gram / (s * s) + diag[:, None, None] * torch.eye(nz, **f64) + dz.t() @ dz
    hinv = torch.cat([torch.cholesky_inverse(torch.linalg.cholesky(part)) for part in hm.split(4096)])
    del hm
    md.gram = None
    wt = md.w.transpose(1, 2)
    one = torch.zeros((p, p), **f64)
    one[:n, :n] = 1.0
    cm = torch.zeros((nt, p, p), **f64)
    cm[:, :n, :n] = mn
    v1, u1 = torch.zeros((nt, p, p), **f64), torch.zeros((nt, p, p), **f64)
    v2, u2 = torch.zeros((3, nz, p, p), **f64), torch.zeros((3, nz, p, p), **f64)
    v3, u3 = torch.zeros((nz, p, p), **f64), torch.zeros((nz, p, p), **f64)
    for _ in range(iters):
        r = v2 - u2
        rz = r[2].clone()
        rz[-1] = 0.0
        back = torch.roll(r[0], 1, 2) - r[0] + torch.roll(r[1], 1, 1) - r[1] - rz
        back[1:] += rz[:-1]
        xh = md.mul(hinv, md.mul(wt, md.fft(v1 - u1)) + md.fft(back + v3 - u3))
        x = md.ifft(xh)
        kx = md.ifft(md.mul(md.w, xh))
        v1 = (cm + rho * (kx + u1)) / (one + rho)
        u1 = u1 + kx - v1
        g = torch.stack([torch.roll(x, -1, 2) - x, torch.roll(x, -1, 1) - x, torch.zeros_like(x)])
        g[2, :-1] = x[1:] - x[:-1]
        g += u2
        v2 = _soft(g, beta / rho)
        u2 = g - v2
        g = x + u3
        v3 = g.clamp_min(0.0) * one
        u3 = g - v3
    return v3[:, :n, :n].contiguous()


def _mux(planes):
    """The 64 x 64 Sylvester Hadamard matrix on every 8 x 8 block of scan points."""
    h = torch.ones((1, 1), device="cuda", dtype=torch.float64)
    while h.shape[0] < 64:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)])
    t, n = planes.shape[0], planes.shape[1]
    b = planes.reshape(t, n // 8, 8, n // 8, 8).permute(0, 1, 3, 2, 4).reshape(-1, 64) @ h
    return b.reshape(t, n // 8, n // 8, 8, 8).permute(0, 1, 3, 2, 4).reshape(t, n, n)


def _exact_fista(case, m):
    md = _Model(case)
    mux = _mux if case["multiplexed"] else (lambda v: v)
    s = md.scale() * (8.0 if case["multiplexed"] else 1.0)
    mn = m.double() / s
    fwd = lambda v: mux(md.forward(v)) / s
    adj = lambda r: md.adjoint(mux(r).contiguous()) / s
    sig = torch.diagonal(md.gram[0]).sqrt()
    thr = (1e-2 * adj(mn).abs().max() * sig / sig.max())[:, None, None]
    x = torch.zeros((case["nz"], case["n"], case["n"]), device="cuda", dtype=torch.float64)
    y, t = x, 1.0
    for _ in range(case["iters"]):
        new = _soft(y - adj(fwd(y) - mn), thr)
        t_new = (1.0 + math.sqrt(1.0 + 4.0 * t * t)) / 2.0
        y, x, t = new + ((t - 1.0) / t_new) * (new - x), new, t_new
    return x.contiguous()


def _conv(x, w, b):
    """3 x 3 x 3 convolution with zero padding, x [ci][z][y][x], w [co][ci][27], one product per tap."""
    _, z, h, v = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    y = b[:, None].expand(-1, z * h * v)
    for t in range(27):
        a, c, e = t // 9, t // 3 % 3, t % 3
        y = y + w[:, :, t] @ xp[:, a:a + z, c:c + h, e:e + v].reshape(x.shape[0], -1)
    return y.reshape(-1, z, h, v)


def _unrolled(md, s, m, theta, stages):
    layers, at = [], 0
    for ci, co in CHANNELS:
        w = theta[at:at + ci * co * 27].reshape(co, ci, 27)
        layers.append((w, theta[at + ci * co * 27:at + ci * co * 27 + co]))
        at += ci * co * 27 + co
    x = torch.zeros((md.case["nz"], md.n, md.n), device="cuda", dtype=torch.float64)
    for k in range(stages):
        r = -m / s if k == 0 else md.forward(x) / s - m / s
        z = x - theta[at + k] * md.adjoint(r) / s
        a = (z / MU0)[None]
        for i, (w, b) in enumerate(layers):
            a = _conv(a, w, b)
            a = torch.relu(a) if i < 3 else a
        x = z + MU0 * a[0]
    return x


def exact(case, seed):
    gen, path = _generator(seed), case["path"]
    batch = case.get("batch", 1)
    if path == "admm_mixed":
        probs = _problems(case)
        return [_exact_admm(p, m, case["iters"]) for p, m in [(p, _measurement(p, gen)) for p in probs]]
    if path == "forward":
        return _Model(case).forward(_volume(case, gen).double()).contiguous()
    if path in ("adjoint", "tikhonov", "admm", "fista"):
        m = _measurement(case, gen)
        if path == "admm":
            return _exact_admm(case, m, case["iters"])
        if path == "fista":
            return _exact_fista(case, m)
        md = _Model(case)
        if path == "adjoint":
            return md.adjoint(m.double()).contiguous()
        return md.tikhonov(m.double(), torch.linalg.cholesky(md.regularised(1e-3))).contiguous()
    if path == "contract":
        nz, nt = case["nz"], case["nt"]
        z = _spectra(case, gen, batch, nz, _volume, (nz + 7) // 8 * 8)
        t = _spectra(case, gen, batch, nt, _measurement, (nt + 7) // 8 * 8)
        w = _table_spectrum(case)
        out_t, out_z = torch.zeros(t.shape, device="cuda", dtype=torch.float64), torch.zeros(z.shape, device="cuda", dtype=torch.float64)
        for v in range(batch):
            out_t[v, :, :nt] = torch.bmm(w, z[v, :, :nz].double())
            out_z[v, :, :nz] = torch.bmm(w.transpose(1, 2), t[v, :, :nt].double())
        return [out_t, out_z]
    m = _stack(_measurement, case, gen, batch)
    md = _Model(case)
    if path == "tikhonov_batch":
        chol = torch.linalg.cholesky(md.regularised(1e-3))
        return torch.stack([md.tikhonov(v.double(), chol) for v in m])
    theta = torch.tensor(_learned_params(case["stages"]), device="cuda", dtype=torch.float64)
    s = md.scale()
    if path == "learned":
        return torch.stack([_unrolled(md, s, v.double(), theta, case["stages"]) for v in m])
    mu = _stack(_volume, case, gen, batch)
    total, theta = 0.0, theta.requires_grad_()
    for v, true in zip(m, mu):
        loss = (((_unrolled(md, s, v.double(), theta, case["stages"]) - true.double()) / MU0) ** 2).mean() / batch
        loss.backward()
        total += float(loss.detach())
    return {"loss": total, "grad": theta.grad.cpu().numpy()}
