// Time-compressed operator.  Every lateral operation of the convolutional
// model (Eq. 11: FFTs, crop, Hadamard multiplexing, the ADMM and FISTA
// updates of the measurement side) acts on all time bins alike, and only
// W_hat mixes them.  The diffusion responses are smooth in time, so W_hat's
// rows span far fewer directions than there are bins: with an orthonormal
// basis Q [nt][r] of that row space
//     W_hat(f) = Q V(f),   V(f) = Q^T W_hat(f)   [r][nz],
// and K^T c = V^T (Q^T c), K x = Q (V x).  The measurement side of every
// solver then works on Q^T m (r planes in place of nt), and only ctof_forward
// expands back to nt bins.
//
// Q is block-diagonal over windows of consecutive bins (each window ends when
// its bin number has doubled or the response has fallen by 1000 within it),
// each with at most 16 columns.  The windows keep the factorisation faithful
// bin by bin and depth by depth, not only in norm.  The rank of a window is
// where the residual, each bin scaled by its DC response and each depth by its
// share of it, falls below 1e-10 and every bin and depth is met to 2e-8 of its
// own DC response.  In FP32 the products Q V must not cancel either: a deep
// layer's response rises by up to eight decades from bin 16 to 32, and a basis in
// the order of size makes its early bins the small difference of large products
// (2.4e-3 of bin 16 for an absorber at 28-32 mm, 1.3e-5 at 20-24 mm).  Where they
// cancel by more than 20 in any bin and depth the basis is turned into the order of
// its bins, and a window that still cancels by more is cut in two.  Emulated in FP32
// every bin and depth then stays within 2e-6, most within 3e-7; a limit of 10 gives
// 5e-7 but up to nine planes more (48 x 48 x 40 x 169: 67 for 60, 80 planes for 64).
// Ranks at 0.5 mm / 25 ps: 67 of 256 bins (128 x 128 scan, 48 depths: 80 planes), 84
// of 512 (64 depths: 96 planes).
// The factorisation is checked on the device over every frequency class and
// is dropped (the handle then works on the nt bins) if it does not hold.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "bulk.cuh"
#include "ctof_internal.h"
#include "time_fit.h"

namespace {

using namespace time_fit;

constexpr int TZ_SAMPLES = 96;       // frequency classes whose rows the basis is fitted on
constexpr int TZ_TILE = 16;          // bins per tile of the expansion

// out[t][s nz + z] = W_hat of class cls[s]
__global__ void k_sample_classes(const double* __restrict__ what64, int nt, int nz, const int* __restrict__ cls,
                                 int ns, double* __restrict__ out) {
  const long long n = (long long)nt * ns * nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int t = (int)(i / (ns * nz)), rem = (int)(i - (long long)t * ns * nz);
    const int s = rem / nz, z = rem - s * nz;
    out[i] = what64[((size_t)cls[s] * nt + t) * nz + z];
  }
}

// One class per block: V = Q^T W_hat (stored FP32 [r][z4], zero padding), and
// the largest |W_hat - Q V| / tol[t][z] over the class, as the bits of a
// non-negative double.
__global__ void __launch_bounds__(256) k_project(const double* __restrict__ what64, int nt, int nz, int z4,
                                                 const double* __restrict__ q, const int4* __restrict__ win, int nwin,
                                                 const double* __restrict__ tol, int rows, float* __restrict__ v32,
                                                 unsigned long long* __restrict__ worst) {
  __shared__ double s_v[TZ_R * 64];
  const int c = blockIdx.x;
  const double* w = what64 + (size_t)c * nt * nz;
  float* out = v32 + (size_t)c * rows * z4;
  double bad = 0.0;
  for (int k = 0; k < nwin; ++k) {
    const int4 g = win[k];  // bins [x, y), first column z, columns w
    for (int i = threadIdx.x; i < g.w * z4; i += blockDim.x) {
      const int j = i / z4, z = i - j * z4;
      double acc = 0.0;
      if (z < nz) {
        for (int t = g.x; t < g.y; ++t) acc = fma(q[(size_t)t * TZ_R + j], w[(size_t)t * nz + z], acc);
        s_v[j * nz + z] = acc;
      }
      out[(size_t)(g.z + j) * z4 + z] = (float)acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (g.y - g.x) * nz; i += blockDim.x) {
      const int t = g.x + i / nz, z = i - (i / nz) * nz;
      double acc = w[(size_t)t * nz + z];
      for (int j = 0; j < g.w; ++j) acc = fma(-q[(size_t)t * TZ_R + j], s_v[j * nz + z], acc);
      bad = fmax(bad, fabs(acc) / tol[t * nz + z]);
    }
    __syncthreads();
  }
  // padding rows of the table
  const int used = win[nwin - 1].z + win[nwin - 1].w;
  for (int i = threadIdx.x; i < (rows - used) * z4; i += blockDim.x) out[(size_t)used * z4 + i] = 0.f;
  for (int o = 16; o > 0; o >>= 1) bad = fmax(bad, __shfl_xor_sync(0xffffffffu, bad, o));
  if ((threadIdx.x & 31) == 0 && bad > 0.0) atomicMax(worst, (unsigned long long)__double_as_longlong(bad));
}

// out[b][r0 + j][p] = sum over the window's bins t of Q[t][j] m[b][t][p].
// m is read once; with up to 16 FMA per value the FMA rate comes next to the
// memory (one volume of 512 bins x 128 x 128: 34 MB, 0.1 GFMA).  Two kernels.
//
// k_compress_bulk (scan points in multiples of 4, 16-byte aligned m): a CTA
// takes 512 / G scan points of one window; the window's rows stream through a
// four-stage ring of bulk copies (8 G rows and their Q rows per stage, 16 KB),
// each thread two points, so that the loads in flight do not depend on the
// registers that the sums need (the register-staged version of this kernel
// took 288 us for 16 volumes of 512 bins x 128 x 128, 537 MB, against 133 us
// here).  G = 4 (few CTAs): four groups of threads split each stage's rows and
// meet in shared memory in a fixed order, which shortens the chain of a
// 100-bin window from 13 stages to 4.
//
// k_compress (anything else): a block takes 32 scan points of one window and
// its eight warps split the window's bins; their sums meet in shared memory in
// a fixed order.
constexpr int CB_PIX = 512, CB_ROWS = 8, CB_STAGES = 4;  // at G = 1
__host__ __device__ constexpr int cb_stage_bytes(int G) { return CB_ROWS * (CB_PIX + G * TZ_R) * 4; }
__host__ __device__ constexpr int cb_smem(int G) { return CB_STAGES * (cb_stage_bytes(G) + 8); }

template <int R, int G>
__device__ __forceinline__ bool compress_window(const float* __restrict__ src, int npix, int pix, int len,
                                                const float* __restrict__ q, int w, float* __restrict__ dst,
                                                unsigned char* sm, int* flag, long long max_polls) {
  constexpr int PIX = CB_PIX / G, ROWS = CB_ROWS * G, SB = cb_stage_bytes(G);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + CB_STAGES * SB);
  const int nst = (len + ROWS - 1) / ROWS;
  auto issue = [&](int s) {  // one warp: a row per lane
    unsigned char* st = sm + (s % CB_STAGES) * SB;
    const int t0 = s * ROWS, nr = min(ROWS, len - t0), r = threadIdx.x;
    uint64_t* b = bar + s % CB_STAGES;
    if (r == 0) {
      bulk::arrive_expect(b, (unsigned)(nr * (pix + TZ_R) * 4));
      bulk::g2s(st + ROWS * PIX * 4, q + (size_t)t0 * TZ_R, nr * TZ_R * 4, b);
    }
    __syncwarp();
    if (r < nr) bulk::g2s(st + r * PIX * 4, src + (size_t)(t0 + r) * npix, pix * 4, b);
  };
  if (threadIdx.x < 32)
    for (int s = 0; s < CB_STAGES && s < nst; ++s) issue(s);
  const int grp = threadIdx.x / (256 / G), pp = threadIdx.x % (256 / G);  // row group, pair of points
  float2 acc[R];
#pragma unroll
  for (int j = 0; j < R; ++j) acc[j] = make_float2(0.f, 0.f);
  for (int s = 0; s < nst; ++s) {
    if (!bulk::block_wait(bar + s % CB_STAGES, (uint32_t)(s / CB_STAGES) & 1u, max_polls)) {
      if (threadIdx.x == 0) {
        atomicOr(flag, 1);
        for (int i = s; i < s + CB_STAGES && i < nst; ++i)
          bulk::wait(bar + i % CB_STAGES, (uint32_t)(i / CB_STAGES) & 1u, bulk::DRAIN_POLLS);
      }
      return false;
    }
    const unsigned char* st = sm + (s % CB_STAGES) * SB;
    const float2* row = reinterpret_cast<const float2*>(st) + pp;
    const float4* qr = reinterpret_cast<const float4*>(st + ROWS * PIX * 4);
    const int nr = min(ROWS, len - s * ROWS);
    auto one = [&](int r) {
      const float2 v = row[r * (PIX / 2)];
#pragma unroll
      for (int j = 0; j < R; j += 4) {
        const float4 c = qr[r * (TZ_R / 4) + j / 4];
        acc[j] = make_float2(fmaf(c.x, v.x, acc[j].x), fmaf(c.x, v.y, acc[j].y));
        acc[j + 1] = make_float2(fmaf(c.y, v.x, acc[j + 1].x), fmaf(c.y, v.y, acc[j + 1].y));
        acc[j + 2] = make_float2(fmaf(c.z, v.x, acc[j + 2].x), fmaf(c.z, v.y, acc[j + 2].y));
        acc[j + 3] = make_float2(fmaf(c.w, v.x, acc[j + 3].x), fmaf(c.w, v.y, acc[j + 3].y));
      }
    };
    if (nr == ROWS) {
#pragma unroll
      for (int r = 0; r < CB_ROWS; ++r) one(G * r + grp);
    } else {
      for (int r = grp; r < nr; r += G) one(r);
    }
    bulk::fence_smem();  // this stage's reads, before the copies that overwrite it
    __syncthreads();
    if (threadIdx.x < 32 && s + CB_STAGES < nst) issue(s + CB_STAGES);
  }
  if constexpr (G > 1) {  // the groups' sums, through the (now idle) first stages
    float2* part = reinterpret_cast<float2*>(sm);
    if (grp > 0) {
#pragma unroll
      for (int j = 0; j < R; ++j) part[((grp - 1) * R + j) * (256 / G) + pp] = acc[j];
    }
    __syncthreads();
    if (grp == 0) {
#pragma unroll
      for (int j = 0; j < R; ++j)
#pragma unroll
        for (int u = 0; u < G - 1; ++u) {
          const float2 o = part[(u * R + j) * (256 / G) + pp];
          acc[j].x += o.x;
          acc[j].y += o.y;
        }
    }
  }
  if (grp == 0 && 2 * pp < pix) {
#pragma unroll
    for (int j = 0; j < R; ++j)
      if (j < w) *reinterpret_cast<float2*>(dst + (size_t)j * npix + 2 * pp) = acc[j];
  }
  return true;
}

template <int G>
__global__ void __launch_bounds__(256, 3) k_compress_bulk(const float* __restrict__ m, int nt, int npix,
                                                          const float* __restrict__ q, const int4* __restrict__ win,
                                                          int nwin, int rows, float* __restrict__ out,
                                                          int* __restrict__ flag, long long max_polls) {
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char csm[];
  // the longest windows come last: start with them
  const int k = nwin - 1 - blockIdx.y;
  const int4 g = win[k];
  const int p0 = blockIdx.x * (CB_PIX / G), pix = min(CB_PIX / G, npix - p0);
  if (threadIdx.x == 0)
    for (int s = 0; s < CB_STAGES; ++s)
      bulk::bar_init(reinterpret_cast<uint64_t*>(csm + CB_STAGES * cb_stage_bytes(G)) + s, 1);
  __syncthreads();
  pdl_wait();
  const float* src = m + ((size_t)blockIdx.z * nt + g.x) * npix + p0;
  float* dst = out + ((size_t)blockIdx.z * rows + g.z) * npix + p0;
  const float* qw = q + (size_t)g.x * TZ_R;
  bool ok;
  if (g.w <= 4)
    ok = compress_window<4, G>(src, npix, pix, g.y - g.x, qw, g.w, dst, csm, flag, max_polls);
  else if (g.w <= 8)
    ok = compress_window<8, G>(src, npix, pix, g.y - g.x, qw, g.w, dst, csm, flag, max_polls);
  else if (g.w <= 12)
    ok = compress_window<12, G>(src, npix, pix, g.y - g.x, qw, g.w, dst, csm, flag, max_polls);
  else
    ok = compress_window<16, G>(src, npix, pix, g.y - g.x, qw, g.w, dst, csm, flag, max_polls);
  if (!ok || k != nwin - 1) return;
  for (int i = threadIdx.x; i < (rows - g.z - g.w) * (CB_PIX / G); i += 256) {  // the planes behind the last window
    const int j = i / (CB_PIX / G), x = i % (CB_PIX / G);
    if (x < pix) dst[(size_t)(g.w + j) * npix + x] = 0.f;
  }
}

__global__ void __launch_bounds__(256) k_compress(const float* __restrict__ m, int nt, int npix,
                                                  const float* __restrict__ q, const int4* __restrict__ win, int nwin,
                                                  int rows, float* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  __shared__ float s_p[8][TZ_R][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int4 g = win[blockIdx.y];
  const int p = blockIdx.x * 32 + lane;
  const float* src = m + (size_t)blockIdx.z * nt * npix + p;
  const bool in = p < npix;
  float acc[TZ_R];
#pragma unroll
  for (int j = 0; j < TZ_R; ++j) acc[j] = 0.f;
  constexpr int U = 8;
  for (int t0 = g.x + warp; t0 < g.y; t0 += 8 * U) {
    float v[U];
#pragma unroll
    for (int i = 0; i < U; ++i) v[i] = in && t0 + 8 * i < g.y ? src[(size_t)(t0 + 8 * i) * npix] : 0.f;
#pragma unroll
    for (int i = 0; i < U; ++i) {
      if (t0 + 8 * i >= g.y) break;
      const float4* row = reinterpret_cast<const float4*>(q + (size_t)(t0 + 8 * i) * TZ_R);
#pragma unroll
      for (int j = 0; j < TZ_R / 4; ++j) {
        const float4 c = __ldg(row + j);
        acc[4 * j] = fmaf(c.x, v[i], acc[4 * j]);
        acc[4 * j + 1] = fmaf(c.y, v[i], acc[4 * j + 1]);
        acc[4 * j + 2] = fmaf(c.z, v[i], acc[4 * j + 2]);
        acc[4 * j + 3] = fmaf(c.w, v[i], acc[4 * j + 3]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < TZ_R; ++j) s_p[warp][j][lane] = acc[j];
  __syncthreads();
  if (!in) return;
  float* dst = out + ((size_t)blockIdx.z * rows + g.z) * npix + p;
  const int end = blockIdx.y == nwin - 1 ? rows - g.z : g.w;  // with the padding planes behind the last window
  for (int j = warp; j < end; j += 8) {
    float s = 0.f;
    if (j < g.w) {
#pragma unroll
      for (int w = 0; w < 8; ++w) s += s_p[w][j][lane];
    }
    dst[(size_t)j * npix] = s;
  }
}

// m[t][p] = sum_j Q[t][j] y[r0 + j][p] for the bins of one tile (up to 16 bins
// of one window): the window's planes are held in registers, the bins written
// as they are formed.  Bound by the writes of m.
template <int V>
__global__ void __launch_bounds__(256) k_expand(const float* __restrict__ y, int npix, const float* __restrict__ q,
                                                const int4* __restrict__ tiles, float* __restrict__ m) {
  pdl_trigger();
  pdl_wait();
  __shared__ float4 s_q[TZ_TILE * TZ_R / 4];
  const int4 g = tiles[blockIdx.y];  // bins [x, y), first column z, columns w
  if ((int)threadIdx.x < (g.y - g.x) * (TZ_R / 4))
    s_q[threadIdx.x] = reinterpret_cast<const float4*>(q + (size_t)g.x * TZ_R)[threadIdx.x];
  const int p = (blockIdx.x * 256 + threadIdx.x) * V;  // V divides npix
  float v[TZ_R][V];
#pragma unroll
  for (int j = 0; j < TZ_R; ++j) {
#pragma unroll
    for (int u = 0; u < V; ++u) v[j][u] = 0.f;
    if (j < g.w && p < npix) {
      const float* src = y + (size_t)(g.z + j) * npix + p;
      if constexpr (V == 2) {
        const float2 f = *reinterpret_cast<const float2*>(src);
        v[j][0] = f.x;
        v[j][V - 1] = f.y;
      } else {
        v[j][0] = *src;
      }
    }
  }
  __syncthreads();
  if (p >= npix) return;
#pragma unroll 4
  for (int t = 0; t < g.y - g.x; ++t) {
    float a[V];
#pragma unroll
    for (int u = 0; u < V; ++u) a[u] = 0.f;
#pragma unroll
    for (int j = 0; j < TZ_R; j += 4) {
      if (j >= g.w) break;
      const float4 c = s_q[t * (TZ_R / 4) + j / 4];
#pragma unroll
      for (int u = 0; u < V; ++u)
        a[u] = fmaf(c.w, v[j + 3][u], fmaf(c.z, v[j + 2][u], fmaf(c.y, v[j + 1][u], fmaf(c.x, v[j][u], a[u]))));
    }
    float* dst = m + (size_t)(g.x + t) * npix + p;
    if constexpr (V == 2)
      *reinterpret_cast<float2*>(dst) = make_float2(a[0], a[V - 1]);
    else
      *dst = a[0];
  }
}

}  // namespace

// Planes the compressed operator works on for a basis of `rank` columns (a
// multiple of 16: the plane tiles of the FFT passes and of the tensor-core
// contractions), or 0 where the nt bins are as cheap: at 48 of 64 planes (config
// 1) a forward call took 32.8 us against 26.6 on the bins.
static int compressed_planes(int nt, int rank) {
  const int rows = ctof_round_up(rank, 16);
  return 2 * rows <= nt ? rows : 0;
}

static ctof_status make_basis(ctof_kernel_s* k, const double* what64, cudaStream_t st) {
  k->tz = nullptr;
  const int nt = k->nt, nz = k->nz;
  if (compressed_planes(nt, TZ_FIRST) == 0) return CTOF_OK;  // too few bins
  // the classes to fit on: the lowest frequencies (DC first) and an even spread of the rest
  std::vector<int> cls;
  for (int i = 0; i < std::min(k->nclass, TZ_SAMPLES / 3); ++i) cls.push_back(i);
  for (int i = 1; i <= TZ_SAMPLES - TZ_SAMPLES / 3; ++i) {
    const int c = (int)((long long)(k->nclass - 1) * i / (TZ_SAMPLES - TZ_SAMPLES / 3));
    if (c > cls.back()) cls.push_back(c);
  }
  const int ns = (int)cls.size();
  std::vector<double> w((size_t)nt * ns * nz);
  struct Buf {
    void* p = nullptr;
    ~Buf() {
      if (p) cudaFree(p);
    }
  } d_cls, d_w, d_q, d_worst;
  // device memory that only the compressed operator needs: without it the handle works on the bins
  auto alloc = [](void** p, size_t bytes) {
    if (cudaMalloc(p, bytes) == cudaSuccess) return true;
    cudaGetLastError();
    *p = nullptr;
    return false;
  };
  if (!alloc(&d_cls.p, cls.size() * sizeof(int)) || !alloc(&d_w.p, w.size() * sizeof(double))) return CTOF_OK;
  CTOF_CUDA_TRY(cudaMemcpyAsync(d_cls.p, cls.data(), cls.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  k_sample_classes<<<152 * 4, 256, 0, st>>>(what64, nt, nz, static_cast<int*>(d_cls.p), ns,
                                            static_cast<double*>(d_w.p));
  CTOF_CUDA_TRY(cudaGetLastError());
  CTOF_CUDA_TRY(cudaMemcpyAsync(w.data(), d_w.p, w.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
  CTOF_CUDA_TRY(cudaStreamSynchronize(st));
  Basis b;
  if (!fit(w, nt, nz, ns, &b)) return CTOF_OK;
  const int rows = compressed_planes(nt, b.rank);
  if (rows == 0) return CTOF_OK;
  std::vector<int4> tiles;
  std::vector<int4> wins;
  for (const Window& g : b.win) {
    wins.push_back(make_int4(g.begin, g.end, g.plane, g.planes));
    for (int t = g.begin; t < g.end; t += TZ_TILE)
      tiles.push_back(make_int4(t, std::min(g.end, t + TZ_TILE), g.plane, g.planes));
  }
  std::vector<float> q32(b.q.size());
  for (size_t i = 0; i < q32.size(); ++i) q32[i] = (float)b.q[i];

  ctof_kernel_s* z = new (std::nothrow) ctof_kernel_s(*k);
  if (!z) return CTOF_ENOMEM;
  z->tz = nullptr;
  z->tz_of = k;
  z->nt = rows;
  z->ldt = rows;
  auto at = [](size_t& off, size_t bytes) {
    off = (off + 255) & ~(size_t)255;
    const size_t o = off;
    off += bytes;
    return o;
  };
  size_t off = 0;
  const size_t wp = contract_warp_floats(rows, nz, 0);
  const size_t wa = wp ? 0 : contract_admm_pipe_floats(rows, nz, 0);
  const size_t ha = wp ? 0 : contract_admm_pipe_floats(rows, nz, 1);
  const size_t o_v = at(off, (size_t)k->nclass * rows * k->z4 * sizeof(float));
  const size_t o_wp = at(off, (size_t)k->nclass * wp * sizeof(float));
  const size_t o_wb = at(off, (size_t)k->nclass * contract_warp_floats(rows, nz, 1) * sizeof(float));
  const size_t o_hb = at(off, (size_t)k->nclass * contract_warp_floats(rows, nz, 2) * sizeof(float));
  const size_t o_wa = at(off, (size_t)k->nclass * wa * sizeof(float));
  const size_t o_ha = at(off, (size_t)k->nclass * ha * sizeof(float));
  const size_t o_q = at(off, q32.size() * sizeof(float));
  const size_t o_win = at(off, wins.size() * sizeof(int4));
  const size_t o_tiles = at(off, tiles.size() * sizeof(int4));
  const size_t o_m = at(off, (size_t)rows * k->n * k->n * sizeof(float));
  z->tz_bytes = off;
  z->d_tz_base = nullptr;
  const size_t qb = b.q.size() * sizeof(double), db = b.tol.size() * sizeof(double);
  if (!alloc(&z->d_tz_base, off) || !alloc(&d_q.p, qb + db) || !alloc(&d_worst.p, sizeof(unsigned long long))) {
    if (z->d_tz_base) cudaFree(z->d_tz_base);
    delete z;
    return CTOF_OK;
  }
  k->tz = z;  // freed with the handle from here on
  char* base = static_cast<char*>(z->d_tz_base);
  z->d_what = reinterpret_cast<float*>(base + o_v);
  z->d_what_pitch = wp ? reinterpret_cast<float*>(base + o_wp) : nullptr;
  z->d_what_block = wp ? reinterpret_cast<float*>(base + o_wb) : nullptr;
  z->d_hinv_block = wp ? reinterpret_cast<float*>(base + o_hb) : nullptr;
  z->d_what_admm = wa ? reinterpret_cast<float*>(base + o_wa) : nullptr;
  z->d_hinv_admm = wa ? reinterpret_cast<float*>(base + o_ha) : nullptr;
  z->d_mstage = reinterpret_cast<float*>(base + o_m);
  z->d_tz_q = reinterpret_cast<float*>(base + o_q);
  z->d_tz_win = reinterpret_cast<int4*>(base + o_win);
  z->d_tz_tiles = reinterpret_cast<int4*>(base + o_tiles);
  z->tz_nwin = (int)wins.size();
  z->tz_ntiles = (int)tiles.size();
  z->tz_nt = nt;
  z->tz_bins = 0;
  for (const Window& g : b.win) {
    if (g.planes < g.end - g.begin) break;
    z->tz_bins = g.end;
  }
  double* d_tol = static_cast<double*>(d_q.p) + b.q.size();
  CTOF_CUDA_TRY(cudaMemcpyAsync(d_q.p, b.q.data(), qb, cudaMemcpyHostToDevice, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(d_tol, b.tol.data(), db, cudaMemcpyHostToDevice, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(z->d_tz_q, q32.data(), q32.size() * sizeof(float), cudaMemcpyHostToDevice, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(z->d_tz_win, wins.data(), wins.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(z->d_tz_tiles, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
  CTOF_CUDA_TRY(cudaMemsetAsync(d_worst.p, 0, sizeof(unsigned long long), st));
  k_project<<<k->nclass, 256, 0, st>>>(what64, nt, nz, k->z4, static_cast<double*>(d_q.p), z->d_tz_win, z->tz_nwin,
                                       d_tol, rows, z->d_what, static_cast<unsigned long long*>(d_worst.p));
  CTOF_CUDA_TRY(cudaGetLastError());
  unsigned long long bits = 0;
  CTOF_CUDA_TRY(cudaMemcpyAsync(&bits, d_worst.p, sizeof(bits), cudaMemcpyDeviceToHost, st));
  CTOF_CUDA_TRY(cudaStreamSynchronize(st));
  double worst;
  memcpy(&worst, &bits, sizeof(worst));
  if (!(worst <= 1.0)) time_basis_free(k);
  return CTOF_OK;
}

ctof_status time_basis_build(ctof_kernel_s* k, const double* what64, cudaStream_t st) {
  try {
    return make_basis(k, what64, st);
  } catch (const std::bad_alloc&) {  // host memory for the fit: the handle works on the bins
    return CTOF_OK;  // (nothing is allocated on the host once k->tz is set)
  }
}

void time_basis_free(ctof_kernel_s* k) {
  ctof_kernel_s* z = k->tz;
  if (!z) return;
  cudaFree(z->d_tz_base);
  delete z;
  k->tz = nullptr;
}

ctof_status time_compress(const ctof_kernel_s* z, int batch, const float* m, float* out, cudaStream_t st) {
  const int npix = z->n * z->n;
  const bool bulk = npix % 4 == 0 && (reinterpret_cast<uintptr_t>(m) & 15) == 0;  // (`out` is the library's own)
  // At G = 1 a CTA takes 512 points of a window: four groups per CTA while there are fewer than two of those per SM.
  // us per call, G = 4 / G = 1: adjoint 64^2 x 48 x 256 (56 CTAs at G = 1) 47.7 / 56.0, 128^2 x 48 x 256 (about 220)
  // 85.6 / 92.8; batched Tikhonov 16 x 64^2 x 32 x 128 (about 500) 228 / 223, 4 x 128^2 x 48 x 256 586 / 578,
  // 16 x 128^2 x 64 x 512 1207 / 1115.
  const bool few = (long long)ctof_div_up(npix, CB_PIX) * z->tz_nwin * batch < 2 * 152;
  auto kern = few ? k_compress_bulk<4> : k_compress_bulk<1>;
  const int smem = few ? cb_smem(4) : cb_smem(1), tile = few ? CB_PIX / 4 : CB_PIX;
  CTOF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  for (int b0 = 0; b0 < batch; b0 += 65535) {
    const int nb = std::min(batch - b0, 65535);
    const float* src = m + (size_t)b0 * z->tz_nt * npix;
    float* dst = out + (size_t)b0 * z->nt * npix;
    if (bulk)
      CTOF_CUDA_TRY(ctof_launch(kern, dim3(ctof_div_up(npix, tile), z->tz_nwin, nb), 256, smem, st, src, z->tz_nt, npix,
                                z->d_tz_q, z->d_tz_win, z->tz_nwin, z->nt, dst, z->d_flags, z->max_polls));
    else
      CTOF_CUDA_TRY(ctof_launch(k_compress, dim3(ctof_div_up(npix, 32), z->tz_nwin, nb), 256, 0, st, src, z->tz_nt,
                                npix, z->d_tz_q, z->d_tz_win, z->tz_nwin, z->nt, dst));
  }
  CTOF_CUDA_TRY(cudaGetLastError());
  return CTOF_OK;
}

ctof_status time_expand(const ctof_kernel_s* z, const float* y, float* m, cudaStream_t st) {
  const int npix = z->n * z->n;
  if (npix % 2 == 0 && (reinterpret_cast<uintptr_t>(m) & 7) == 0)
    CTOF_CUDA_TRY(ctof_launch(k_expand<2>, dim3(ctof_div_up(npix, 512), z->tz_ntiles), 256, 0, st, y, npix, z->d_tz_q,
                              z->d_tz_tiles, m));
  else
    CTOF_CUDA_TRY(ctof_launch(k_expand<1>, dim3(ctof_div_up(npix, 256), z->tz_ntiles), 256, 0, st, y, npix, z->d_tz_q,
                              z->d_tz_tiles, m));
  CTOF_CUDA_TRY(cudaGetLastError());
  return CTOF_OK;
}
