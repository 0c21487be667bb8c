// Single-volume contractions of small class blocks, one warp per frequency
// class (Eq. 11 in the lateral Fourier domain, and the ADMM x-update on it):
//   FWD   out[t] = sum_z W[t][z] x[z]
//   ADJ   out[z] = sum_t W[t][z] c[t]
//   TIK   out[z] = sum_j H[j][z] (W^T c)[j]                 (H symmetric)
//   ADMM  b = W^T c / s + s_hat - L x,  x += H b,  Kx = W x / s
// for the complex vectors of the up-to-four frequencies that share the real
// block W [nt][nz] of their class (8 real right-hand sides).
//
// A time-compressed block is 15 KB (80 planes x 48 depths): too little work
// for a thread block, whose barriers between the phases cost more than the
// phases.  Launch times with a thread block / a warp per class: forward at
// 256 x 256 x 32 x 128 (48 planes) 162 / 47 us (42 us of HBM time for what it
// reads and writes), adjoint at 128 x 128 x 48 x 256 (80 planes) 76 / 37 us (20),
// x-update there 97 / 70 us (42 us for 287 MB; 73 us before the depth blocks
// became a template parameter).  Here a CTA (one per SM) holds a ring of
// shared-memory slots filled by bulk asynchronous copies, one class per slot,
// and each of its warps takes every NW-th class through all phases by itself:
// no block barrier, the warps drift apart and their phases overlap.  The warp
// that finishes a class refills its slot with the class that follows a ring's
// length later, so up to NS classes (200 KB) are in flight per SM.
//
// Arithmetic is FP32 FMA (the x-update: TF32 tensor-core products in three terms,
// as in contract_admm.cu).  Adjoint passes give a lane one 16-byte chunk of a
// row and one of 32/q interleaved row sets, for all eight right-hand sides, so
// each word of the block is read once; the row sets meet in the warp's scratch.
// Forward passes give a lane whole rows (row pitch 4 (q | 1) words: 16-byte
// reads of eight rows fall on distinct banks).  Vector reads are uniform over
// a row set (broadcast).
//
// Every wait is bounded: a warp whose wait runs out sets the handle's sticky
// flag and stops; the CTA then waits, with its own limit, for the copies it
// still has in flight.
#include <cuda_runtime.h>

#include "bulk.cuh"
#include "ctof_internal.h"
#include "tf32_mma.cuh"

namespace {

enum { WM_FWD = 0, WM_ADJ = 1, WM_TIK = 2, WM_ADMM = 3 };

constexpr int WARP_SMEM = 227 * 1024;
constexpr int MAX_WARPS = 12;
constexpr int MAX_PAIRS = 8;  // ADMM: 16 warps of up to 128 registers

// Partials of an adjoint pass: 16-byte units (members 2h, 2h + 1 of depth 4 k + a
// of row set j) at (2 a + h) PART_PITCH + j q + k, so that both the lanes that
// write them and the eight depths x four members that read them fall on
// distinct banks.
constexpr int PART_PITCH = 33;
constexpr int PART_BYTES = 8 * PART_PITCH * 16;

struct WarpPlan {
  int nt, nz, z4, q, sw;         // q = z4 / 4 chunks per row, sw = row pitch of the W table (floats)
  int J;                         // row sets of an adjoint pass
  int tb, zb;                    // 8-row blocks of t and z (ADMM's block layout)
  int cs, zs;                    // member pitch (complex) of T and Z vectors
  int nw, ns;                    // warps, slots
  int o_h, o_c, o_s, o_x, o_hdr, slot;  // byte offsets in a slot, its size
  int o_b, scratch;              // warp scratch: [partials][vector], bytes
  int o_scr, o_bar, total;
  unsigned w_bytes, h_bytes, c_bytes, v_bytes;
};

inline int rup(int x, int m) { return (x + m - 1) / m * m; }

WarpPlan plan_for(int mode, int nt, int nz, int nw) {
  WarpPlan P{};
  P.nt = nt;
  P.nz = nz;
  P.z4 = rup(nz, 4);
  P.q = P.z4 / 4;
  P.sw = 4 * (P.q | 1);
  P.J = 32 / P.q;
  P.tb = rup(nt, 8) / 8;
  P.zb = rup(nz, 8) / 8;
  // ADMM reads vector fragments at (member pitch) g/2 + row tg: 8 banks apart
  P.cs = mode == WM_ADMM ? rup(8 * P.tb, 16) + 4 : rup(nt, 2);
  P.zs = mode == WM_ADMM ? rup(8 * P.zb, 16) + 4 : rup(P.z4, 2);
  P.w_bytes = (unsigned)(mode == WM_ADMM ? P.tb * P.zb * 256 : nt * P.sw * 4);
  P.h_bytes = mode == WM_ADMM ? (unsigned)(P.zb * P.zb * 256) : mode == WM_TIK ? (unsigned)(nz * P.z4 * 4) : 0;
  P.c_bytes = (unsigned)(rup(nt, 2) * 8);
  P.v_bytes = (unsigned)(rup(nz, 2) * 8);
  P.o_h = rup((int)P.w_bytes, 16);
  P.o_c = P.o_h + rup((int)P.h_bytes, 16);
  P.o_s = P.o_c + (mode == WM_FWD ? 0 : 4 * P.cs * 8);
  P.o_x = P.o_s + (mode == WM_ADMM ? 4 * P.zs * 8 : 0);
  P.o_hdr = P.o_x + (mode == WM_FWD || mode == WM_ADMM ? 4 * P.zs * 8 : 0);
  P.slot = rup(P.o_hdr + 32, 128);
  P.o_b = mode == WM_FWD || mode == WM_ADMM ? 0 : PART_BYTES;
  P.scratch = rup(P.o_b + (mode == WM_TIK ? 4 * P.zs * 8 : mode == WM_ADMM ? 2 * 8 * P.zb * 32 : 0), 128);
  P.nw = nw;
  P.o_scr = 0;
  const int fixed = nw * P.scratch + 16 * 64 + 128;
  P.ns = (WARP_SMEM - fixed) / P.slot;
  if (P.ns > 32) P.ns = 32;
  P.o_bar = 0;  // set below
  P.total = 0;
  if (P.ns >= 1) {
    P.o_scr = P.ns * P.slot;
    P.o_bar = P.o_scr + nw * P.scratch;
    P.total = P.o_bar + P.ns * 16;
  }
  return P;
}

// As many warps (up to 12) as have a slot each and one more in flight.
// Blocks so large that fewer than four warps find room keep the CTA-wide
// kernels.
bool choose_plan(int mode, int nt, int nz, WarpPlan* out) {
  if (nz > 64) return false;
  for (int nw = mode == WM_ADMM ? MAX_PAIRS : MAX_WARPS; nw >= 4; --nw) {
    const WarpPlan P = plan_for(mode, nt, nz, nw);
    if (P.ns > nw) {
      *out = P;
      return true;
    }
  }
  return false;
}

struct WarpArgs {
  WarpPlan P;
  const float* w;        // [nclass][nt][sw]; ADMM: [nclass][tb][zb][64]
  const float* h;        // [nclass][nz][z4]; ADMM: [nclass][zb][zb][64]
  const float* lap;      // [nclass]
  const int* members;    // [nclass][4]
  int nclass;
  const float2* in;      // FWD: Z spectra, otherwise T spectra
  const float2* s_hat;   // ADMM
  float2* x_hat;         // ADMM: in / out; ADJ, TIK: out
  float2* out_t;         // FWD, ADMM
  int ldt, ldz;
  float inv_s;
};

__device__ __forceinline__ void cfma(float2& acc, float w, float x, float y) {
  acc.x = fmaf(w, x, acc.x);
  acc.y = fmaf(w, y, acc.y);
}

// Partials over row set j of sum M[r][z] v[m][r], one lane per (j, chunk);
// sets take contiguous even-sized runs of rows.
__device__ __forceinline__ void adj_pass(const WarpPlan& P, const float* M, int pitch, int rows, const float2* v,
                                         int vpitch, float2* part, int lane) {
  const int j = lane / P.q, k = lane - j * P.q;
  if (j < P.J) {
    float2 acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[a][m] = make_float2(0.f, 0.f);
    const int per = ((rows + P.J - 1) / P.J + 1) & ~1;
    const int r0 = j * per, r1 = min(rows, r0 + per);
    const float* mp = M + 4 * k;
    // sums of eight rows, then their sum: FP32 rounding of the solves that follow a
    // W^T c comes from this accumulation (1.7e-6 against 2.0e-6 in one run of 32 rows)
    for (int rb = r0; rb < r1; rb += 8) {
      const int re = min(r1, rb + 8);
      float2 t[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int m = 0; m < 4; ++m) t[a][m] = make_float2(0.f, 0.f);
      int r = rb;
#pragma unroll 2
      for (; r + 2 <= re; r += 2) {
        const float4 w0 = *reinterpret_cast<const float4*>(mp + r * pitch);
        const float4 w1 = *reinterpret_cast<const float4*>(mp + (r + 1) * pitch);
        float4 c[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) c[m] = *reinterpret_cast<const float4*>(v + m * vpitch + r);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          cfma(t[0][m], w0.x, c[m].x, c[m].y);
          cfma(t[1][m], w0.y, c[m].x, c[m].y);
          cfma(t[2][m], w0.z, c[m].x, c[m].y);
          cfma(t[3][m], w0.w, c[m].x, c[m].y);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          cfma(t[0][m], w1.x, c[m].z, c[m].w);
          cfma(t[1][m], w1.y, c[m].z, c[m].w);
          cfma(t[2][m], w1.z, c[m].z, c[m].w);
          cfma(t[3][m], w1.w, c[m].z, c[m].w);
        }
      }
      if (r < re) {
        const float4 w0 = *reinterpret_cast<const float4*>(mp + r * pitch);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float2 c = v[m * vpitch + r];
          cfma(t[0][m], w0.x, c.x, c.y);
          cfma(t[1][m], w0.y, c.x, c.y);
          cfma(t[2][m], w0.z, c.x, c.y);
          cfma(t[3][m], w0.w, c.x, c.y);
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[a][m] = cadd(acc[a][m], t[a][m]);
    }
    float4* dst = reinterpret_cast<float4*>(part) + lane;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      dst[(2 * a) * PART_PITCH] = make_float4(acc[a][0].x, acc[a][0].y, acc[a][1].x, acc[a][1].y);
      dst[(2 * a + 1) * PART_PITCH] = make_float4(acc[a][2].x, acc[a][2].y, acc[a][3].x, acc[a][3].y);
    }
  }
  __syncwarp();
}

// Sum of the row sets' partials for (z, m).
__device__ __forceinline__ float2 adj_sum(const WarpPlan& P, const float2* part, int z, int m) {
  const float2* u = part + 2 * ((2 * (z & 3) + (m >> 1)) * PART_PITCH + (z >> 2)) + (m & 1);
  float2 s = u[0];
  for (int j = 1; j < P.J; ++j) {
    const float2 p = u[2 * j * P.q];
    s.x += p.x;
    s.y += p.y;
  }
  return s;
}

// out[f_m][t] = sum_z W[t][z] x[m][z], two rows per lane at a time.
// x entries z in [nz, z4) are zero.
__device__ __forceinline__ void fwd_pass(const WarpPlan& P, const float* W, const float2* x, int xpitch,
                                         const int (&mem)[4], float2* __restrict__ out, int ld, int lane) {
  for (int t0 = lane; t0 < P.nt; t0 += 64) {
    const bool two = t0 + 32 < P.nt;
    const float* wa = W + t0 * P.sw;
    const float* wb = two ? wa + 32 * P.sw : wa;
    float2 a[4], b[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) a[m] = b[m] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int k = 0; k < P.q; ++k) {
      const float4 u = *reinterpret_cast<const float4*>(wa + 4 * k);
      const float4 v = *reinterpret_cast<const float4*>(wb + 4 * k);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float u0 = h ? u.z : u.x, u1 = h ? u.w : u.y, v0 = h ? v.z : v.x, v1 = h ? v.w : v.y;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float4 c = *reinterpret_cast<const float4*>(x + m * xpitch + 4 * k + 2 * h);
          cfma(a[m], u0, c.x, c.y);
          cfma(b[m], v0, c.x, c.y);
          cfma(a[m], u1, c.z, c.w);
          cfma(b[m], v1, c.z, c.w);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (mem[m] < 0) continue;
      out[(size_t)mem[m] * ld + t0] = a[m];
      if (two) out[(size_t)mem[m] * ld + t0 + 32] = b[m];
    }
  }
}

// One lane: class c (members f) into a slot, completing on `full`: the header and
// the class's tables first, then its vectors.
template <int MODE>
__device__ __forceinline__ void fill_tables(const WarpArgs& A, int c, int4 f, float dl, unsigned char* st,
                                            uint64_t* full) {
  const WarpPlan& P = A.P;
  const int present = (f.x >= 0) + (f.y >= 0) + (f.z >= 0) + (f.w >= 0);
  const unsigned per = MODE == WM_FWD ? P.v_bytes : P.c_bytes + (MODE == WM_ADMM ? 2 * P.v_bytes : 0);
  *reinterpret_cast<int4*>(st + P.o_hdr) = f;
  if (MODE == WM_ADMM) *reinterpret_cast<float*>(st + P.o_hdr + 16) = dl;
  bulk::arrive_expect(full, P.w_bytes + P.h_bytes + present * per);
  bulk::g2s(st, A.w + (size_t)c * (P.w_bytes >> 2), P.w_bytes, full);
  if (MODE >= WM_TIK) bulk::g2s(st + P.o_h, A.h + (size_t)c * (P.h_bytes >> 2), P.h_bytes, full);
}

template <int MODE>
__device__ __forceinline__ void fill_vectors(const WarpArgs& A, int4 f4, unsigned char* st, uint64_t* full) {
  const WarpPlan& P = A.P;
  const int f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (f[m] < 0) continue;
    if (MODE == WM_FWD) {
      bulk::g2s(st + P.o_x + m * P.zs * 8, A.in + (size_t)f[m] * A.ldz, P.v_bytes, full);
    } else {
      bulk::g2s(st + P.o_c + m * P.cs * 8, A.in + (size_t)f[m] * A.ldt, P.c_bytes, full);
    }
    if (MODE == WM_ADMM) {
      bulk::g2s(st + P.o_s + m * P.zs * 8, A.s_hat + (size_t)f[m] * A.ldz, P.v_bytes, full);
      bulk::g2s(st + P.o_x + m * P.zs * 8, A.x_hat + (size_t)f[m] * A.ldz, P.v_bytes, full);
    }
  }
}

template <int MODE>
__device__ __forceinline__ void do_class(const WarpArgs& A, unsigned char* st, unsigned char* scr, int lane) {
  const WarpPlan& P = A.P;
  const float* W = reinterpret_cast<const float*>(st);
  const float* H = reinterpret_cast<const float*>(st + P.o_h);
  const float2* C = reinterpret_cast<const float2*>(st + P.o_c);
  float2* X = reinterpret_cast<float2*>(st + P.o_x);
  const int4 f4 = *reinterpret_cast<const int4*>(st + P.o_hdr);
  const int mem[4] = {f4.x, f4.y, f4.z, f4.w};
  float2* part = reinterpret_cast<float2*>(scr);
  float2* vec = reinterpret_cast<float2*>(scr + P.o_b);
  const int g = lane >> 2, mm = lane & 3;  // element-wise phases: depth 8 i + g of member mm
  const int fm = mm == 0 ? f4.x : mm == 1 ? f4.y : mm == 2 ? f4.z : f4.w;
  if (MODE == WM_FWD) {
    // entries past nz come from the row's padding: zero them (the table's padding columns are zero too)
    if (P.nz + g < P.z4 && g < 4) X[mm * P.zs + P.nz + g] = make_float2(0.f, 0.f);
    __syncwarp();
    fwd_pass(P, W, X, P.zs, mem, A.out_t, A.ldt, lane);
    return;
  }
  adj_pass(P, W, P.sw, P.nt, C, P.cs, part, lane);
  if (MODE == WM_ADJ) {
    if (fm >= 0)
      for (int z = g; z < P.nz; z += 8) A.x_hat[(size_t)fm * A.ldz + z] = adj_sum(P, part, z, mm);
    return;
  }
  if (MODE == WM_TIK) {
    for (int z = g; z < P.nz; z += 8) vec[mm * P.zs + z] = adj_sum(P, part, z, mm);
    __syncwarp();
    adj_pass(P, H, P.z4, P.nz, vec, P.zs, part, lane);
    if (fm >= 0)
      for (int z = g; z < P.nz; z += 8) A.x_hat[(size_t)fm * A.ldz + z] = adj_sum(P, part, z, mm);
    return;
  }
}

// dh + dl += A B in 3xTF32 (the small products in their own accumulator).
__device__ __forceinline__ void mma_3x(float (&dh)[4], float (&dl)[4], const float (&a)[4], const unsigned (&b)[4]) {
  unsigned ah[4], al[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split_fast(a[i], ah[i], al[i]);
  mma_tf32(dl, al, b[0], b[1]);
  mma_tf32(dl, ah, b[2], b[3]);
  mma_tf32(dh, ah, b[0], b[1]);
}

// Barrier `id` over the two warps of a pair.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool pair_any(int id, bool v) {
  int out;
  asm volatile(
      "{\n"
      ".reg .pred q, p;\n"
      "setp.ne.s32 q, %2, 0;\n"
      "bar.red.or.pred p, %1, 64, q;\n"
      "selp.s32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(out)
      : "r"(id), "r"((int)v)
      : "memory");
  return out != 0;
}

// The ADMM x-update of one class by a pair of warps (a 28 KB slot leaves room
// for seven classes on an SM, and seven single warps are too few to cover the
// latency of this chain: 77 us against 73), its three products on the
// warp-level tensor-core MMA (m16n8k8: N = the eight right-hand sides) as
// 3xTF32.  W and H come in 8 x 8 blocks whose 64 words are permuted so that
// fragments of the block and of its transpose load without bank conflicts:
//   word(i, j) = 32 (j / 4) + 4 ((i + 4 (j / 4)) mod 8) + j mod 4.
// Lane (g, tg) holds rows g and g + 8 of member tg in every result.  The first
// two products split their K steps between the warps, which exchange half of
// the partial sums: warp `half` finishes rows 8 half + g of every 16-row tile;
// the third splits the t tiles.
template <int ZB>
__device__ __forceinline__ void do_admm(const WarpArgs& A, const unsigned char* st, float* vec, int half, int bar,
                                        int lane) {
  const WarpPlan& P = A.P;
  const int g = lane >> 2, tg = lane & 3, hg = g >> 2;
  const int offF0 = 4 * g + tg, offF2 = 32 + 4 * ((g + 4) & 7) + tg;  // (row g, columns tg, tg + 4)
  const int offA0 = 32 * hg + 4 * ((tg + 4 * hg) & 7) + (g & 3);      // (row tg, column g)
  const int offA2 = 32 * hg + 4 * ((tg + 4 + 4 * hg) & 7) + (g & 3);  // (row tg + 4, column g)
  constexpr int MZ = (ZB + 1) / 2;  // 16-row z tiles
  const int TB = P.tb, nt = P.nt, nz = P.nz;
  const float* W = reinterpret_cast<const float*>(st);
  const float* H = reinterpret_cast<const float*>(st + P.o_h);
  const float* C = reinterpret_cast<const float*>(st + P.o_c) + (g >> 1) * 2 * P.cs + (g & 1);
  const int4 f4 = *reinterpret_cast<const int4*>(st + P.o_hdr);
  const float dl = *reinterpret_cast<const float*>(st + P.o_hdr + 16);
  const int fm = tg == 0 ? f4.x : tg == 1 ? f4.y : tg == 2 ? f4.z : f4.w;
  float dh[MZ][4], dlo[MZ][4];
#pragma unroll
  for (int mt = 0; mt < MZ; ++mt)
#pragma unroll
    for (int i = 0; i < 4; ++i) dh[mt][i] = dlo[mt][i] = 0.f;
  // ---- y = W^T c ----
#pragma unroll 2
  for (int ks = half; ks < TB; ks += 2) {
    const int t = 8 * ks + tg;
    unsigned b[4];
    split_fast(t < nt ? C[2 * t] : 0.f, b[0], b[2]);
    split_fast(t + 4 < nt ? C[2 * t + 8] : 0.f, b[1], b[3]);
    const float* w = W + ks * ZB * 64;
#pragma unroll
    for (int mt = 0; mt < MZ; ++mt) {
      const bool up = 2 * mt + 1 < ZB;
      const float* wl = w + 2 * mt * 64;
      const float a[4] = {wl[offA0], up ? wl[64 + offA0] : 0.f, wl[offA2], up ? wl[64 + offA2] : 0.f};
      mma_3x(dh[mt], dlo[mt], a, b);
    }
  }
  float* xch = vec + 64 * ZB;  // [z][8] partial sums handed to the other warp
  auto give = [&]() {          // rows that the other warp finishes
#pragma unroll
    for (int mt = 0; mt < MZ; ++mt) {
      const int z = 16 * mt + 8 * (1 - half) + g;
      const float2 v = half ? make_float2(dh[mt][0] + dlo[mt][0], dh[mt][1] + dlo[mt][1])
                            : make_float2(dh[mt][2] + dlo[mt][2], dh[mt][3] + dlo[mt][3]);
      if (z < 8 * ZB) *reinterpret_cast<float2*>(xch + z * 8 + 2 * tg) = v;
    }
  };
  auto take = [&](int mt) {  // this warp's row of tile mt, both partial sums
    const int z = 16 * mt + 8 * half + g;
    const float2 o = *reinterpret_cast<const float2*>(xch + z * 8 + 2 * tg);
    const float2 v = half ? make_float2(dh[mt][2] + dlo[mt][2], dh[mt][3] + dlo[mt][3])
                          : make_float2(dh[mt][0] + dlo[mt][0], dh[mt][1] + dlo[mt][1]);
    return make_float2(v.x + o.x, v.y + o.y);
  };
  give();
  pair_sync(bar);
  // ---- b = y / s + s_hat - L x,  L = dl I + Dz^T Dz ----
  const float2* S = reinterpret_cast<const float2*>(st + P.o_s) + tg * P.zs;
  const float2* X = reinterpret_cast<const float2*>(st + P.o_x) + tg * P.zs;
#pragma unroll
  for (int mt = 0; mt < MZ; ++mt) {
    const int z = 16 * mt + 8 * half + g;
    if (z >= 8 * ZB) continue;
    float2 b = make_float2(0.f, 0.f);
    if (z < nz) {
      const float2 y = take(mt), xz = X[z], s = S[z];
      float2 lx = make_float2(dl * xz.x, dl * xz.y);
      if (z > 0) {
        const float2 p = X[z - 1];
        lx.x += xz.x - p.x;
        lx.y += xz.y - p.y;
      }
      if (z < nz - 1) {
        const float2 n = X[z + 1];
        lx.x -= n.x - xz.x;
        lx.y -= n.y - xz.y;
      }
      b = make_float2(y.x * A.inv_s + s.x - lx.x, y.y * A.inv_s + s.y - lx.y);
    }
    *reinterpret_cast<float2*>(vec + z * 8 + 2 * tg) = b;
  }
  pair_sync(bar);
  // ---- x += H b ----
#pragma unroll
  for (int mt = 0; mt < MZ; ++mt)
#pragma unroll
    for (int i = 0; i < 4; ++i) dh[mt][i] = dlo[mt][i] = 0.f;
#pragma unroll
  for (int kk = 0; kk < MZ; ++kk) {
    const int ks = 2 * kk + half;
    if (ks >= ZB) break;  // (odd ZB: the second warp has one step less)
    unsigned b[4];
    split_fast(vec[(8 * ks + tg) * 8 + g], b[0], b[2]);
    split_fast(vec[(8 * ks + tg + 4) * 8 + g], b[1], b[3]);
#pragma unroll
    for (int mt = 0; mt < MZ; ++mt) {
      const bool up = 2 * mt + 1 < ZB;
      const float* h = H + (2 * mt * ZB + ks) * 64;
      const float a[4] = {h[offF0], up ? h[ZB * 64 + offF0] : 0.f, h[offF2], up ? h[ZB * 64 + offF2] : 0.f};
      mma_3x(dh[mt], dlo[mt], a, b);
    }
  }
  give();  // (the partial sums of y were taken before the barrier above)
  pair_sync(bar);
#pragma unroll
  for (int mt = 0; mt < MZ; ++mt) {
    const int z = 16 * mt + 8 * half + g;
    if (z >= 8 * ZB) continue;
    float2 xn = make_float2(0.f, 0.f);
    if (z < nz) {
      const float2 d = take(mt), xz = X[z];
      xn = make_float2(xz.x + d.x, xz.y + d.y);
      if (fm >= 0) A.x_hat[(size_t)fm * A.ldz + z] = xn;
    }
    *reinterpret_cast<float2*>(vec + z * 8 + 2 * tg) = xn;
  }
  pair_sync(bar);
  // ---- Kx = W x / s, two 16-row tiles at a time ----
  unsigned xb[ZB][4];
#pragma unroll
  for (int ks = 0; ks < ZB; ++ks) {
    split_fast(vec[(8 * ks + tg) * 8 + g], xb[ks][0], xb[ks][2]);
    split_fast(vec[(8 * ks + tg + 4) * 8 + g], xb[ks][1], xb[ks][3]);
  }
  float2* dst = fm >= 0 ? A.out_t + (size_t)fm * A.ldt : nullptr;
  for (int r0 = 4 * half; r0 < TB; r0 += 8) {
    float eh[2][4], el[2][4];
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int i = 0; i < 4; ++i) eh[v][i] = el[v][i] = 0.f;
    const float* w = W + (size_t)r0 * ZB * 64;
    const bool b1 = r0 + 1 < TB, b2 = r0 + 2 < TB, b3 = r0 + 3 < TB;
#pragma unroll
    for (int ks = 0; ks < ZB; ++ks) {
      const float* q = w + ks * 64;
      const float a0[4] = {q[offF0], b1 ? q[ZB * 64 + offF0] : 0.f, q[offF2], b1 ? q[ZB * 64 + offF2] : 0.f};
      mma_3x(eh[0], el[0], a0, xb[ks]);
      if (b2) {
        const float* q2 = q + 2 * ZB * 64;
        const float a1[4] = {q2[offF0], b3 ? q2[ZB * 64 + offF0] : 0.f, q2[offF2], b3 ? q2[ZB * 64 + offF2] : 0.f};
        mma_3x(eh[1], el[1], a1, xb[ks]);
      }
    }
    if (dst) {
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = 8 * (r0 + 2 * v + u) + g;
          if (t < nt)
            dst[t] = make_float2((eh[v][2 * u] + el[v][2 * u]) * A.inv_s,
                                 (eh[v][2 * u + 1] + el[v][2 * u + 1]) * A.inv_s);
        }
    }
  }
}

// Fill number `n` (1, 2, ...) of a slot was issued: published by the lane that
// issued it.  A warp waits for this before it waits on the slot's barrier: the
// barrier alone cannot tell "fill n has not been issued, fill n - 1 is still in
// flight" (a warp can be a whole ring ahead of a slower one) from "done".
__device__ __forceinline__ void publish(int* issued, int n) {
  asm volatile("st.release.cta.shared::cta.s32 [%0], %1;\n" ::"r"(bulk::saddr(issued)), "r"(n) : "memory");
}
__device__ __forceinline__ int published(const int* issued) {
  int n;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];\n" : "=r"(n) : "r"(bulk::saddr(issued)) : "memory");
  return n;
}
__device__ __forceinline__ bool wait_fill(uint64_t* full, const int* issued, int n, long long max_polls) {
  long long i = 0;
  for (; i < max_polls && published(issued) < n; ++i) {
  }
  if (i == max_polls) return false;
  return bulk::wait(full, (uint32_t)(n - 1) & 1u, max_polls);
}

// ZB: 8-row z blocks of the ADMM products (ceil(nz / 8)).
template <int MODE, int ZB>
__global__ void __launch_bounds__(MODE == WM_ADMM ? MAX_PAIRS * 64 : MAX_WARPS * 32, 1)
    k_contract_warp(const __grid_constant__ WarpArgs A, int* __restrict__ flag, long long max_polls) {
  extern __shared__ __align__(128) unsigned char wsm[];
  pdl_trigger();
  const WarpPlan& P = A.P;
  // worker: the warp or pair of warps that takes every NW-th class; its first lane fills slots
  constexpr int WT = MODE == WM_ADMM ? 64 : 32;
  const int worker = threadIdx.x / WT, lane = threadIdx.x & 31;
  const bool first = threadIdx.x % WT == 0;
  const int NW = P.nw, NS = P.ns;
  uint64_t* full = reinterpret_cast<uint64_t*>(wsm + P.o_bar);
  int* issued = reinterpret_cast<int*>(full + NS);  // fills issued per slot
  const int mine = (int)blockIdx.x < A.nclass ? (A.nclass - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  // (the slots need no zeroing: what an absent member's vector holds only reaches results that are not stored)
  if (threadIdx.x < NS) {
    bulk::bar_init(full + threadIdx.x, 1);
    issued[threadIdx.x] = 0;
  }
  __syncthreads();
  auto cls = [&](int k) { return (int)blockIdx.x + k * (int)gridDim.x; };
  auto header = [&](int k, int4& f, float& dl) {
    f = __ldg(reinterpret_cast<const int4*>(A.members) + cls(k));
    dl = MODE == WM_ADMM ? __ldg(A.lap + cls(k)) + 1.0f : 0.f;
  };
  // the first ring, slot s by worker s mod NW: the tables do not depend on earlier work in the stream
  if (first) {
    int4 f;
    float dl;
    for (int k = worker; k < NS && k < mine; k += NW) {
      header(k, f, dl);
      fill_tables<MODE>(A, cls(k), f, dl, wsm + k * P.slot, full + k);
    }
    pdl_wait();
    for (int k = worker; k < NS && k < mine; k += NW) {
      fill_vectors<MODE>(A, *reinterpret_cast<const int4*>(wsm + k * P.slot + P.o_hdr), wsm + k * P.slot, full + k);
      publish(issued + k, 1);
    }
  }
  __syncwarp();
  pdl_wait();
  for (int k = worker; k < mine; k += NW) {
    const int s = k % NS, kn = k + NS;
    int4 fn = make_int4(-1, -1, -1, -1);
    float dn = 0.f;
    if (first && kn < mine) header(kn, fn, dn);  // the refill's, ahead of its use
    const bool late = !wait_fill(full + s, issued + s, k / NS + 1, max_polls);
    if (MODE == WM_ADMM ? pair_any(1 + worker, late) : __any_sync(0xffffffffu, late)) {
      if (first) atomicOr(flag, 1);
      break;
    }
    unsigned char* scr = wsm + P.o_scr + worker * P.scratch;
    if constexpr (MODE == WM_ADMM)
      do_admm<ZB>(A, wsm + s * P.slot, reinterpret_cast<float*>(scr), (threadIdx.x >> 5) & 1, 1 + worker, lane);
    else
      do_class<MODE>(A, wsm + s * P.slot, scr, lane);
    bulk::fence_smem();  // the worker's accesses of the slot, before the copies into it
    if constexpr (MODE == WM_ADMM)
      pair_sync(1 + worker);
    else
      __syncwarp();
    if (first && kn < mine) {
      fill_tables<MODE>(A, cls(kn), fn, dn, wsm + s * P.slot, full + s);
      fill_vectors<MODE>(A, fn, wsm + s * P.slot, full + s);
      publish(issued + s, kn / NS + 1);
    }
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < NS && issued[threadIdx.x] > 0)  // (at once unless a worker gave up)
    bulk::wait(full + threadIdx.x, (uint32_t)(issued[threadIdx.x] - 1) & 1u, bulk::DRAIN_POLLS);
}

// W_hat rows at the pitch sw: out[row][sw] (zero padding).
__global__ void k_pitch_rows(const float* __restrict__ in, long long rows, int nz, int z4, int sw,
                             float* __restrict__ out) {
  const long long n = rows * sw;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / sw;
    const int z = (int)(i - r * sw);
    out[i] = z < nz ? in[r * z4 + z] : 0.f;
  }
}

template <int MODE, int ZB>
ctof_status launch(const ctof_kernel_s* k, const WarpPlan& P, WarpArgs& A, cudaStream_t st) {
  A.P = P;
  A.w = MODE == WM_ADMM ? k->d_what_block : k->d_what_pitch;
  A.lap = k->d_lap;
  A.members = k->d_members;
  A.nclass = k->nclass;
  A.ldt = k->ldt;
  A.ldz = k->ldz;
  auto kern = k_contract_warp<MODE, ZB>;
  CTOF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, P.total));
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, k->device);
  const int grid = k->nclass < nsm ? k->nclass : nsm;
  const int threads = P.nw * (MODE == WM_ADMM ? 64 : 32);
  CTOF_CUDA_TRY(ctof_launch(kern, grid, threads, P.total, st, A, k->d_flags, k->max_polls));
  CTOF_CUDA_TRY(cudaGetLastError());
  return CTOF_OK;
}

}  // namespace

// Each mode has sizes of its own: rows at the odd pitch and the partials of an adjoint pass take more
// room than the x-update's blocks (8 depths: the x-update fits to 688 planes, the adjoint to 535, the
// Tikhonov solve to 528).  Where a mode has no room, the CTA-per-class kernel takes the call.
bool contract_warp_takes(const ctof_kernel_s* k, WarpCall call) {
  WarpPlan P;
  const int mode = call == WarpCall::Forward ? WM_FWD : call == WarpCall::Adjoint ? WM_ADJ : WM_TIK;
  return k->d_what_pitch && choose_plan(mode, k->nt, k->nz, &P);
}

int contract_warp_slots(int nt, int nz) {
  WarpPlan P;
  return choose_plan(WM_ADMM, nt, nz, &P) ? P.ns : 0;
}

size_t contract_warp_floats(int nt, int nz, int which) {
  WarpPlan P;
  if (!choose_plan(WM_ADMM, nt, nz, &P)) return 0;
  return which == 0 ? (size_t)nt * P.sw : (which == 1 ? P.w_bytes : P.h_bytes) / 4;
}

ctof_status contract_warp_prepare(const ctof_kernel_s* k, cudaStream_t st) {
  if (!k->d_what_pitch) return CTOF_OK;
  const int sw = 4 * ((k->z4 / 4) | 1);
  k_pitch_rows<<<152 * 8, 256, 0, st>>>(k->d_what, (long long)k->nclass * k->nt, k->nz, k->z4, sw, k->d_what_pitch);
  const int tb = rup(k->nt, 8) / 8, zb = rup(k->nz, 8) / 8;
  k_block_rows<<<152 * 8, 256, 0, st>>>(k->d_what, k->nt, k->nz, k->z4, tb, zb, k->d_what_block, k->nclass);
  k_block_rows<<<152 * 8, 256, 0, st>>>(k->d_hinv, k->nz, k->nz, k->z4, zb, zb, k->d_hinv_block, k->nclass);
  CTOF_CUDA_TRY(cudaGetLastError());
  return CTOF_OK;
}

ctof_status contract_warp_forward(const ctof_kernel_s* k, const float2* in_z, float2* out_t, cudaStream_t st) {
  WarpPlan P;
  if (!k->d_what_pitch || !choose_plan(WM_FWD, k->nt, k->nz, &P)) return CTOF_EUNSUPPORTED;
  WarpArgs A{};
  A.in = in_z;
  A.out_t = out_t;
  return launch<WM_FWD, 1>(k, P, A, st);
}

ctof_status contract_warp_adjoint(const ctof_kernel_s* k, const float2* in_t, float2* out_z, cudaStream_t st) {
  WarpPlan P;
  if (!k->d_what_pitch || !choose_plan(WM_ADJ, k->nt, k->nz, &P)) return CTOF_EUNSUPPORTED;
  WarpArgs A{};
  A.in = in_t;
  A.x_hat = out_z;
  return launch<WM_ADJ, 1>(k, P, A, st);
}

ctof_status contract_warp_tikhonov(const ctof_kernel_s* k, const float* hinv, const float2* m_hat, float2* x_hat,
                                   cudaStream_t st) {
  WarpPlan P;
  if (!k->d_what_pitch || !choose_plan(WM_TIK, k->nt, k->nz, &P)) return CTOF_EUNSUPPORTED;
  WarpArgs A{};
  A.h = hinv;
  A.in = m_hat;
  A.x_hat = x_hat;
  return launch<WM_TIK, 1>(k, P, A, st);
}

ctof_status contract_warp_admm(const ctof_kernel_s* k, const float2* c_hat, const float2* s_hat, float2* x_hat,
                               float2* kx_hat, float inv_scale, cudaStream_t st) {
  WarpPlan P;
  if (!k->d_what_pitch || !choose_plan(WM_ADMM, k->nt, k->nz, &P)) return CTOF_EUNSUPPORTED;
  WarpArgs A{};
  A.h = k->d_hinv_block;
  A.in = c_hat;
  A.s_hat = s_hat;
  A.x_hat = x_hat;
  A.out_t = kx_hat;
  A.inv_s = inv_scale;
  switch ((k->nz + 7) / 8) {
    case 1: return launch<WM_ADMM, 1>(k, P, A, st);
    case 2: return launch<WM_ADMM, 2>(k, P, A, st);
    case 3: return launch<WM_ADMM, 3>(k, P, A, st);
    case 4: return launch<WM_ADMM, 4>(k, P, A, st);
    case 5: return launch<WM_ADMM, 5>(k, P, A, st);
    case 6: return launch<WM_ADMM, 6>(k, P, A, st);
    case 7: return launch<WM_ADMM, 7>(k, P, A, st);
    default: return launch<WM_ADMM, 8>(k, P, A, st);
  }
}
