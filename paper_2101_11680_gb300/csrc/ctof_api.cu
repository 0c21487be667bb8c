// C ABI entry points: argument validation, the handle and its workspaces, and
// the orchestration of the forward / adjoint / reconstruction chains.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "ctof_internal.h"

static thread_local char g_last_error[512] = "";

void ctof_set_last_cuda_error(cudaError_t e, const char* what, const char* file, int line) {
  snprintf(g_last_error, sizeof(g_last_error), "%s (%s) at %s:%d: %s", cudaGetErrorName(e), what, file, line,
           cudaGetErrorString(e));
}

void ctof_set_last_error_text(const char* msg) { snprintf(g_last_error, sizeof(g_last_error), "%s", msg); }

namespace {


bool finite_pos(double v) { return isfinite(v) && v > 0.0; }

int next_pow2(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

ctof_status validate(const ctof_optics* o, const ctof_grid* g) {
  if (!o || !g) return CTOF_EINVAL;
  if (!(isfinite(o->mua_mm) && o->mua_mm >= 0.0) || !finite_pos(o->musp_mm) || !(isfinite(o->n) && o->n >= 1.0))
    return CTOF_EINVAL;
  if (!isfinite(o->z0_mm)) return CTOF_EINVAL;
  if (g->nx <= 0 || g->ny <= 0 || g->nz <= 0 || g->nt <= 0) return CTOF_EINVAL;
  if (!finite_pos(g->dx_mm) || !finite_pos(g->dy_mm) || !finite_pos(g->dz_mm) || !finite_pos(g->z_first_mm) ||
      !finite_pos(g->dt_ps))
    return CTOF_EINVAL;
  if (g->conv_mode != CTOF_LINEAR && g->conv_mode != CTOF_CIRCULAR) return CTOF_EINVAL;
  if (g->nx != g->ny) return CTOF_EUNSUPPORTED;
  if (g->nz > 64 || g->nt > 1024) return CTOF_EUNSUPPORTED;
  // one frequency class (W_hat block, vectors, partial sums) must fit in shared memory
  {
    const size_t admm = contract_admm_smem_bytes(g->nt, g->nz, 1);
    const size_t other = contract_smem_bytes(g->nt, g->nz);
    if (admm > 227 * 1024 || other > 227 * 1024) return CTOF_EUNSUPPORTED;
  }
  if (g->conv_mode == CTOF_LINEAR) {
    if (g->nx < 4 || g->nx > 256) return CTOF_EUNSUPPORTED;
  } else {
    if (g->nx < 32 || g->nx > 512 || (g->nx & (g->nx - 1)) != 0) return CTOF_EUNSUPPORTED;
  }
  return CTOF_OK;
}

// Frequency classes: half-plane frequencies with equal W_hat.  The kernel is
// even in x and y (and symmetric under x <-> y when dx == dy), so W_hat(kx,ky)
// depends on (kx, |ky|) -- and on the unordered pair when symmetric.
void make_classes(int P, bool symmetric, std::vector<int>& members, std::vector<float>& lap) {
  const int h = P / 2 + 1;
  const int A = h;
  std::vector<int> key_to_class((size_t)A * A, -1);
  std::vector<std::pair<int, int>> keys;
  // enumerate keys in (b, a) order so that class 0 is the DC frequency
  for (int b = 0; b < A; ++b)
    for (int a = 0; a < A; ++a) {
      if (symmetric && a > b) continue;
      key_to_class[(size_t)b * A + a] = (int)keys.size();
      keys.push_back({a, b});
    }
  const int nclass = (int)keys.size();
  members.assign((size_t)nclass * 4, -1);
  std::vector<int> count(nclass, 0);
  for (int ky = 0; ky < P; ++ky)
    for (int kx = 0; kx < h; ++kx) {
      int a = kx, b = ky <= P / 2 ? ky : P - ky;
      if (symmetric && a > b) std::swap(a, b);
      const int c = key_to_class[(size_t)b * A + a];
      const int f = ky * h + kx;
      members[(size_t)c * 4 + count[c]++] = f;
    }
  // the class's first member must be (kx = a, |ky| = b) for the table gather
  for (int c = 0; c < nclass; ++c) {
    const int a = keys[c].first, b = keys[c].second;
    for (int m = 0; m < count[c]; ++m) {
      const int f = members[(size_t)c * 4 + m];
      const int kx = f % h, ky = f / h;
      if (kx == a && (ky == b || ky == (P - b) % P)) {
        std::swap(members[(size_t)c * 4], members[(size_t)c * 4 + m]);
        break;
      }
    }
  }
  lap.resize(nclass);
  const double pi = 3.14159265358979323846;
  for (int c = 0; c < nclass; ++c) {
    const double sa = sin(pi * keys[c].first / P), sb = sin(pi * keys[c].second / P);
    lap[c] = (float)(4.0 * sa * sa + 4.0 * sb * sb);
  }
}

struct Carver {
  size_t off = 0;
  template <typename T>
  size_t take(size_t count) {
    off = (off + 255) & ~(size_t)255;
    const size_t at = off;
    off += count * sizeof(T);
    return at;
  }
};

ctof_status forward_impl(ctof_kernel_s* k, const float* mu, float* m, cudaStream_t st) {
  CTOF_TRY(fft_forward_planes(k, mu, k->nz, k->n, k->n, k->n, k->d_inter_z, k->d_spec_z, k->ldz, st));
  CTOF_TRY(contract_forward(k, k->d_spec_z, k->d_spec_t, st));
  return fft_inverse_planes(k, k->d_spec_t, k->ldt, k->nt, k->n, k->n, k->d_inter_t, m, k->n, st);
}

ctof_status adjoint_impl(ctof_kernel_s* k, const float* m, float* vol, cudaStream_t st) {
  CTOF_TRY(fft_forward_planes(k, m, k->nt, k->n, k->n, k->n, k->d_inter_t, k->d_spec_t, k->ldt, st));
  CTOF_TRY(contract_adjoint(k, k->d_spec_t, k->d_spec_z, st));
  return fft_inverse_planes(k, k->d_spec_z, k->ldz, k->nz, k->n, k->n, k->d_inter_z, vol, k->n, st);
}

// Measurement m [nt][n][n] (device memory) into `out` as the planes that
// operator o works on: Q^T m for a time-compressed one, a copy otherwise.
ctof_status stage_measurement(const ctof_kernel_s* o, const float* m, float* out, cudaStream_t st) {
  if (o->tz_nt) return time_compress(o, 1, m, out, st);
  CTOF_CUDA_TRY(cudaMemcpyAsync(out, m, (size_t)o->nt * o->n * o->n * sizeof(float), cudaMemcpyDeviceToDevice, st));
  return CTOF_OK;
}

// The operator that a solver runs on.
ctof_kernel_s* solver_ops(ctof_kernel_s* k, const ctof_solver_params* prm) {
  return prm->solver == CTOF_SOLVER_TIKHONOV ? ctof_ops_once(k) : ctof_ops(k);
}

// m = A mu in all nt bins, with `mux` y = S A mu (S acts on all bins alike, so
// before the expansion).
ctof_status forward_bins(ctof_kernel_s* k, const float* mu, float* m, bool mux, cudaStream_t st) {
  ctof_kernel_s* o = ctof_ops_once(k);
  float* planes = o->tz_nt ? o->d_u1 : m;
  CTOF_TRY(forward_impl(o, mu, planes, st));
  if (mux) CTOF_TRY(block_hadamard(planes, o->nt, o->n, st));
  return o->tz_nt ? time_expand(o, planes, m, st) : CTOF_OK;
}

// ADMM set-up on the staged measurement d_mstage: the TV weight and the state reset.
ctof_status admm_setup(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st) {
  const int nt = k->nt, nz = k->nz, n = k->n, P = k->p;
  const size_t pp = (size_t)P * P;
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_scalars, 0, 16 * sizeof(double), st));
  if (prm->tv_beta < 0) {
    CTOF_TRY(adjoint_impl(k, k->d_mstage, k->d_vstage, st));
    CTOF_TRY(reduce_max_abs(k->d_vstage, (size_t)nz * n * n, k->d_scalars + 1, st));
  }
  CTOF_TRY(admm_set_beta(k->d_scalars, prm->tv_beta, prm->beta_rel, 1.0 / (k->scale * k->scale), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_spec_t2, 0, (size_t)k->nf * k->ldt * sizeof(float2), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_spec_z, 0, (size_t)k->nf * k->ldz * sizeof(float2), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_spec_z2, 0, (size_t)k->nf * k->ldz * sizeof(float2), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_u1, 0, (size_t)nt * n * n * sizeof(float), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_u2a, 0, 3 * nz * pp * sizeof(float), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_u3, 0, nz * pp * sizeof(float), st));
  return CTOF_OK;
}

// The x-update of iteration `it` (per frequency class) and K x.
ctof_status admm_contract(ctof_kernel_s* k, cudaStream_t st) {
  return contract_admm(k, k->d_spec_t2, k->d_spec_z, k->d_spec_z2, k->d_spec_t, (float)(1.0 / k->scale), st);
}

// T side of an iteration (not after the last): K x -> v1/u1 -> c_hat.
ctof_status admm_t_side(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st) {
  CTOF_TRY(fft_cols_inverse(k, k->d_spec_t, k->ldt, k->nt, k->n, k->d_inter_t, st));
  CTOF_TRY(fft_rows_admm_t(k, k->d_inter_t, k->d_mstage, k->d_u1, (float)(1.0 / k->scale), (float)prm->rho, st));
  return fft_cols_forward(k, k->d_inter_t, k->nt, k->n, k->d_spec_t2, k->ldt, st);
}

// Z side of iteration `it`: x -> TV / nonnegativity prox -> s_hat (the last
// iteration writes the crop of v3 to d_vstage instead).
ctof_status admm_z_side(ctof_kernel_s* k, const ctof_solver_params* prm, int it, cudaStream_t st) {
  const int nz = k->nz, P = k->p;
  const float rho = (float)prm->rho;
  const bool last = it == prm->iters - 1;
  float* u2[2] = {k->d_u2a, k->d_u2b};
  CTOF_TRY(fft_cols_inverse(k, k->d_spec_z2, k->ldz, nz, P, k->d_inter_z, st));
  CTOF_TRY(fft_rows_inverse(k, k->d_inter_z, nz, P, P, k->d_xs, P, st));
  CTOF_TRY(admm_tv_stencil(k, k->d_xs, u2[it & 1], u2[(it + 1) & 1], k->d_u3, k->d_s, k->d_scalars, rho,
                           last ? k->d_vstage : nullptr, st));
  if (!last) {
    CTOF_TRY(fft_rows_forward(k, k->d_s, nz, P, P, P, k->d_inter_z, st));
    CTOF_TRY(fft_cols_forward(k, k->d_inter_z, nz, P, k->d_spec_z, k->ldz, st));
  }
  return CTOF_OK;
}

// The rest of iteration `it` after the x-update, one side after the other;
// `ev_mid` (optional) is recorded between the two.
ctof_status admm_side(ctof_kernel_s* k, const ctof_solver_params* prm, int it, cudaStream_t st, cudaEvent_t ev_mid) {
  if (it != prm->iters - 1) CTOF_TRY(admm_t_side(k, prm, st));
  if (ev_mid) CTOF_CUDA_TRY(cudaEventRecordWithFlags(ev_mid, st, cudaEventRecordExternal));
  return admm_z_side(k, prm, it, st);
}

// A branch of a captured graph: `side` runs from where `st` is at fork() until join().
struct GraphBranch {
  cudaStream_t side = nullptr;
  cudaEvent_t ev = nullptr;
  ~GraphBranch() {
    if (ev) cudaEventDestroy(ev);
    if (side) cudaStreamDestroy(side);
  }
  ctof_status make() {
    CTOF_CUDA_TRY(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    CTOF_CUDA_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    return CTOF_OK;
  }
  ctof_status order(cudaStream_t first, cudaStream_t then) {
    CTOF_CUDA_TRY(cudaEventRecord(ev, first));
    CTOF_CUDA_TRY(cudaStreamWaitEvent(then, ev, 0));
    return CTOF_OK;
  }
};

// ADMM on the staged measurement d_mstage; result (crop of v3) in d_vstage.
// The two sides of an iteration touch different state and neither fills the
// chip alone (short chains of latency-bound passes), so they run as two
// branches of the graph (one after the other when the stages are timed).
ctof_status admm_enqueue(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st, bool timed) {
  CTOF_TRY(admm_setup(k, prm, st));
  if (!(timed && k->timing)) {
    GraphBranch br;
    CTOF_TRY(br.make());
    for (int it = 0; it < prm->iters; ++it) {
      CTOF_TRY(admm_contract(k, st));
      if (it == prm->iters - 1) return admm_z_side(k, prm, it, st);
      CTOF_TRY(br.order(st, br.side));
      CTOF_TRY(admm_t_side(k, prm, br.side));
      CTOF_TRY(admm_z_side(k, prm, it, st));
      CTOF_TRY(br.order(br.side, st));
    }
    return CTOF_OK;
  }
  cudaEvent_t* ev = (timed && k->timing) ? k->events : nullptr;
  for (int it = 0; it < prm->iters; ++it) {
    if (ev) CTOF_CUDA_TRY(cudaEventRecordWithFlags(ev[4 * it + 0], st, cudaEventRecordExternal));
    CTOF_TRY(admm_contract(k, st));
    if (ev) CTOF_CUDA_TRY(cudaEventRecordWithFlags(ev[4 * it + 1], st, cudaEventRecordExternal));
    CTOF_TRY(admm_side(k, prm, it, st, ev ? ev[4 * it + 2] : nullptr));
    if (ev) CTOF_CUDA_TRY(cudaEventRecordWithFlags(ev[4 * it + 3], st, cudaEventRecordExternal));
  }
  return CTOF_OK;
}

void destroy_events(ctof_kernel_s* k) {
  for (int i = 0; i < k->n_events; ++i) cudaEventDestroy(k->events[i]);
  delete[] k->events;
  k->events = nullptr;
  k->n_events = 0;
}

ctof_status ensure_events(ctof_kernel_s* k, int count) {
  if (k->n_events >= count) return CTOF_OK;
  destroy_events(k);
  k->events = new (std::nothrow) cudaEvent_t[count];
  if (!k->events) return CTOF_ENOMEM;
  for (int i = 0; i < count; ++i) {
    if (cudaEventCreate(&k->events[i]) != cudaSuccess) {
      k->n_events = i;
      destroy_events(k);
      return CTOF_ECUDA;
    }
  }
  k->n_events = count;
  return CTOF_OK;
}

// Autotuner: times each column-pass tile (32 columns of 8 or 16 planes, 16
// columns of 8 or 16 planes) on the handle's own buffers for the four
// column-pass shapes of an ADMM iteration and keeps the fastest.
// Synchronous; must run outside stream capture.
ctof_status autotune(ctof_kernel_s* k, cudaStream_t st) {
  if (k->tuned) return CTOF_OK;
  // tile codes: 8 / 16 planes in 32-column tiles, 100 + 8 / 16 in 16-column tiles
  const int cands[4] = {8, 16, 108, 116};
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  CTOF_CUDA_TRY(cudaEventCreate(&e0));
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return CTOF_ECUDA;
  }
  ctof_status s = CTOF_OK;
  const int n = k->n, P = k->p;
  if (cudaMemsetAsync(k->d_inter_t, 0, fft_inter_elems(k, k->nt, n) * sizeof(float2), st) != cudaSuccess ||
      cudaMemsetAsync(k->d_inter_z, 0, fft_inter_elems(k, k->nz, P) * sizeof(float2), st) != cudaSuccess ||
      cudaMemsetAsync(k->d_spec_t, 0, (size_t)k->nf * k->ldt * sizeof(float2), st) != cudaSuccess ||
      cudaMemsetAsync(k->d_spec_z2, 0, (size_t)k->nf * k->ldz * sizeof(float2), st) != cudaSuccess)
    s = CTOF_ECUDA;
  for (int use = 0; use < 4 && s == CTOF_OK; ++use) {
    float best_ms = 1e30f;
    int best = 16;
    for (int ci = 0; ci < 4 && s == CTOF_OK; ++ci) {
      const int pb = cands[ci];
      auto launch = [&]() -> ctof_status {
        switch (use) {
          case 0: return fft_cols_forward_pb(k, k->d_inter_t, k->nt, n, k->d_spec_t2, k->ldt, pb, st);
          case 1: return fft_cols_inverse_pb(k, k->d_spec_t, k->ldt, k->nt, n, k->d_inter_t, pb, st);
          case 2: return fft_cols_forward_pb(k, k->d_inter_z, k->nz, P, k->d_spec_z, k->ldz, pb, st);
          default: return fft_cols_inverse_pb(k, k->d_spec_z2, k->ldz, k->nz, P, k->d_inter_z, pb, st);
        }
      };
      s = launch();
      if (s != CTOF_OK) break;
      if (cudaEventRecord(e0, st) != cudaSuccess) { s = CTOF_ECUDA; break; }
      for (int r = 0; r < 3 && s == CTOF_OK; ++r) s = launch();
      if (s != CTOF_OK) break;
      float ms = 0.f;
      if (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
          cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
        s = CTOF_ECUDA;
        break;
      }
      if (ms < best_ms) {
        best_ms = ms;
        best = pb;
      }
    }
    k->tune_pb[use] = best;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (s == CTOF_OK) k->tuned = 1;
  return s;
}

// The handle's ADMM graph for these parameters (captured on first use; `st`
// only serves the autotuner).
ctof_status admm_graph(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st) {
  CTOF_TRY(autotune(k, st));
  const bool same = k->graph && k->graph_iters == prm->iters && k->graph_rho == prm->rho &&
                    k->graph_beta == prm->tv_beta && k->graph_beta_rel == prm->beta_rel &&
                    k->graph_timing == k->timing && k->graph_polls == k->max_polls &&
                    std::equal(k->graph_pb, k->graph_pb + 4, k->tune_pb);
  if (!same) {
    if (k->graph) {
      cudaGraphExecDestroy(k->graph);
      k->graph = nullptr;
    }
    if (k->timing) CTOF_TRY(ensure_events(k, 4 * prm->iters));
    cudaStream_t cap = nullptr;
    CTOF_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) {
      cudaStreamDestroy(cap);
      CTOF_CUDA_TRY(e);
    }
    const ctof_status s = admm_enqueue(k, prm, cap, true);
    e = cudaStreamEndCapture(cap, &g);
    cudaStreamDestroy(cap);
    if (s != CTOF_OK) {
      if (g) cudaGraphDestroy(g);
      return s;
    }
    CTOF_CUDA_TRY(e);
    {
      size_t nn = 0;
      int kernels = 0;
      if (cudaGraphGetNodes(g, nullptr, &nn) == cudaSuccess && nn > 0) {
        std::vector<cudaGraphNode_t> nodes(nn);
        if (cudaGraphGetNodes(g, nodes.data(), &nn) == cudaSuccess)
          for (size_t i = 0; i < nn; ++i) {
            cudaGraphNodeType t;
            if (cudaGraphNodeGetType(nodes[i], &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) ++kernels;
          }
      }
      k->graph_kernel_nodes = kernels;
    }
    e = cudaGraphInstantiate(&k->graph, g, 0);
    cudaGraphDestroy(g);
    CTOF_CUDA_TRY(e);
    k->graph_timing = k->timing;
    k->graph_polls = k->max_polls;
    std::copy(k->tune_pb, k->tune_pb + 4, k->graph_pb);
    k->graph_iters = prm->iters;
    k->graph_rho = prm->rho;
    k->graph_beta = prm->tv_beta;
    k->graph_beta_rel = prm->beta_rel;
  }
  return CTOF_OK;
}

ctof_status admm_run(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st) {
  CTOF_TRY(admm_graph(k, prm, st));
  CTOF_CUDA_TRY(cudaGraphLaunch(k->graph, st));
  return CTOF_OK;
}

}  // namespace

ctof_status tikhonov_inverse(ctof_kernel_s* k, double lambda, const float** hinv, cudaStream_t st) {
  if (!(lambda > 0.0) || !isfinite(lambda)) return CTOF_EINVAL;
  k = ctof_owner(k);
  int slot = k->tik_lambda[0] == lambda ? 0 : (k->tik_lambda[1] == lambda ? 1 : -1);
  if (slot < 0) {
    slot = 1 - k->tik_last;  // replace the slot not used last
    if (!k->d_tik_hinv[slot]) {
      void* p = nullptr;
      if (cudaMalloc(&p, (size_t)k->nclass * k->nz * k->z4 * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        return CTOF_ENOMEM;
      }
      k->d_tik_hinv[slot] = static_cast<float*>(p);
    }
    k->tik_lambda[slot] = -1.0;
    CTOF_TRY(build_tikhonov_factors(k, slot, lambda, st));
  }
  k->tik_last = slot;
  *hinv = k->d_tik_hinv[slot];
  return CTOF_OK;
}

namespace {

ctof_status tikhonov_run(ctof_kernel_s* k, const ctof_solver_params* prm, cudaStream_t st, double* lambda_out) {
  const double lambda = prm->tik_lambda_rel * k->gram_max;
  const float* hinv = nullptr;
  CTOF_TRY(tikhonov_inverse(k, lambda, &hinv, st));
  *lambda_out = lambda;
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_scalars, 0, 16 * sizeof(double), st));
  CTOF_TRY(fft_forward_planes(k, k->d_mstage, k->nt, k->n, k->n, k->n, k->d_inter_t, k->d_spec_t, k->ldt, st));
  CTOF_TRY(contract_tikhonov(k, hinv, k->d_spec_t, k->d_spec_z, st));
  return fft_inverse_planes(k, k->d_spec_z, k->ldz, k->nz, k->n, k->n, k->d_inter_z, k->d_vstage, k->n, st);
}

// FISTA for Eq. 10 on the staged measurement (result in d_vstage).  Normalised
// units (A_n = A / s, step 1); lam0 by the same rule as the ADMM TV weight;
// lam(z) follows the DC depth sensitivity.  With `mux` the operator is the
// composite S A of Eq. 12 (S = H_64 on every 8 x 8 block of scan points, so
// the normalisation is 8 s) and the staged measurement is the multiplexed y.
// S S = 64, so the gradient A^T S (S A x - y) = A^T (64 A x - S y) takes S once,
// on the measurement.
// Eight launches per iteration: neither the residual nor the gradient exists as
// an array of its own, the row passes form them between the two transforms of
// a row (fourteen launches of 3 to 9 us each before, mostly latency).
// Workspace: ADMM state buffers.
ctof_status fista_run(ctof_kernel_s* k, const ctof_solver_params* prm, bool mux, cudaStream_t st) {
  const size_t vol = (size_t)k->nz * k->n * k->n;
  float* y = k->d_u3;
  float* x = k->d_xs;
  float* lam = k->d_u2a;
  const double sc = k->scale * (mux ? 8.0 : 1.0);
  const float inv_s2 = (float)(1.0 / (sc * sc));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_scalars, 0, 16 * sizeof(double), st));
  if (mux) CTOF_TRY(block_hadamard(k->d_mstage, k->nt, k->n, st));
  if (prm->tv_beta < 0) {
    CTOF_TRY(adjoint_impl(k, k->d_mstage, k->d_vstage, st));
    CTOF_TRY(reduce_max_abs(k->d_vstage, vol, k->d_scalars + 1, st));
  }
  CTOF_TRY(admm_set_beta(k->d_scalars, prm->tv_beta, prm->beta_rel, 1.0 / (sc * sc), st));
  CTOF_TRY(fista_lambda(k, k->d_scalars, lam, st));
  CTOF_CUDA_TRY(cudaMemsetAsync(y, 0, vol * sizeof(float), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(x, 0, vol * sizeof(float), st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_inter_z, 0, fft_inter_elems(k, k->nz, k->n) * sizeof(float2), st));
  double t = 1.0;
  for (int it = 0; it < prm->iters; ++it) {
    CTOF_TRY(fft_cols_forward(k, k->d_inter_z, k->nz, k->n, k->d_spec_z, k->ldz, st));
    CTOF_TRY(contract_forward(k, k->d_spec_z, k->d_spec_t, st));
    CTOF_TRY(fft_cols_inverse(k, k->d_spec_t, k->ldt, k->nt, k->n, k->d_inter_t, st));
    CTOF_TRY(fft_rows_resid_t(k, k->d_inter_t, k->d_mstage, mux ? 64.f : 1.f, st));
    CTOF_TRY(fft_cols_forward(k, k->d_inter_t, k->nt, k->n, k->d_spec_t, k->ldt, st));
    CTOF_TRY(contract_adjoint(k, k->d_spec_t, k->d_spec_z, st));
    CTOF_TRY(fft_cols_inverse(k, k->d_spec_z, k->ldz, k->nz, k->n, k->d_inter_z, st));
    const double t_next = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
    CTOF_TRY(fft_rows_fista(k, k->d_inter_z, y, x, lam, inv_s2, (float)((t - 1.0) / t_next), st));
    t = t_next;
  }
  CTOF_CUDA_TRY(cudaMemcpyAsync(k->d_vstage, x, vol * sizeof(float), cudaMemcpyDeviceToDevice, st));
  return CTOF_OK;
}

ctof_status validate_params(const ctof_solver_params* p) {
  if (!p) return CTOF_EINVAL;
  if (p->solver == CTOF_SOLVER_FISTA_L1 || p->solver == CTOF_SOLVER_FISTA_L1_MUX) {
    if (p->iters < 1 || p->iters > 100000) return CTOF_EINVAL;
    if (!isfinite(p->tv_beta)) return CTOF_EINVAL;
    if (p->tv_beta < 0 && !(isfinite(p->beta_rel) && p->beta_rel >= 0)) return CTOF_EINVAL;
    return CTOF_OK;
  }
  if (p->solver == CTOF_SOLVER_ADMM_TV) {
    if (p->iters < 1 || p->iters > 100000) return CTOF_EINVAL;
    if (!finite_pos(p->rho)) return CTOF_EINVAL;
    if (!isfinite(p->tv_beta)) return CTOF_EINVAL;
    if (p->tv_beta < 0 && !(isfinite(p->beta_rel) && p->beta_rel >= 0)) return CTOF_EINVAL;
    return CTOF_OK;
  }
  if (p->solver == CTOF_SOLVER_TIKHONOV) return finite_pos(p->tik_lambda_rel) ? CTOF_OK : CTOF_EINVAL;
  return CTOF_EINVAL;
}

// Runs the chosen solver on d_mstage, leaving the result in d_vstage.
ctof_status solve_staged(ctof_kernel_s* k, const ctof_solver_params* prm, double* lambda, cudaStream_t st) {
  *lambda = 0.0;
  if (prm->solver == CTOF_SOLVER_ADMM_TV) return admm_run(k, prm, st);
  if (prm->solver == CTOF_SOLVER_FISTA_L1) return fista_run(k, prm, false, st);
  if (prm->solver == CTOF_SOLVER_FISTA_L1_MUX) {
    if (k->n % 8 != 0) return CTOF_EUNSUPPORTED;
    return fista_run(k, prm, true, st);
  }
  return tikhonov_run(k, prm, st, lambda);
}

}  // namespace

ctof_status take_device_status(ctof_kernel_s* k, cudaStream_t st) {
  int flag = 0;
  CTOF_CUDA_TRY(cudaMemcpyAsync(&flag, k->d_flags, sizeof(int), cudaMemcpyDeviceToHost, st));
  CTOF_CUDA_TRY(cudaMemsetAsync(k->d_flags, 0, sizeof(int), st));
  CTOF_CUDA_TRY(cudaStreamSynchronize(st));
  return flag ? CTOF_ETIMEOUT : CTOF_OK;
}

namespace {

// Synchronising report: parameters used, a NaN/Inf scan of the result, and
// the handle's sticky device status (a bounded wait that ran out).
ctof_status fill_report(ctof_kernel_s* k, const ctof_solver_params* prm, double lambda, ctof_report* rep,
                        cudaStream_t st) {
  int* flag = reinterpret_cast<int*>(k->d_scalars + 8);
  CTOF_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int), st));
  CTOF_TRY(check_finite(k->d_vstage, (size_t)k->nz * k->n * k->n, flag, st));
  double sc[10];
  CTOF_CUDA_TRY(cudaMemcpyAsync(sc, k->d_scalars, 10 * sizeof(double), cudaMemcpyDeviceToHost, st));
  CTOF_CUDA_TRY(cudaStreamSynchronize(st));
  int bad = 0;
  memcpy(&bad, &sc[8], sizeof(int));
  const ctof_status waits = take_device_status(k, st);
  rep->scale = k->scale;
  rep->beta = prm->solver == CTOF_SOLVER_TIKHONOV ? 0.0 : sc[0];
  rep->lambda = lambda;
  rep->iters_done = prm->solver == CTOF_SOLVER_TIKHONOV ? 1 : prm->iters;
  if (waits != CTOF_OK) return waits;
  return bad ? CTOF_ENONFINITE : CTOF_OK;
}

// ADMM on `count` handles at once: every problem runs its own graph (kept with
// its handle, independent of the callers' buffers, and shared with
// ctof_reconstruct) on a stream of its own that starts where `st` is; `st`
// goes on when all are done.
ctof_status batch_run(int count, const ctof_kernel* ks, const float* const* d_m, const ctof_solver_params* prm,
                      float* const* d_mu, cudaStream_t st) {
  for (int i = 0; i < count; ++i) {
    ctof_kernel_s* o = ctof_ops(ks[i]);
    if (!o->batch_stream) CTOF_CUDA_TRY(cudaStreamCreateWithFlags(&o->batch_stream, cudaStreamNonBlocking));
    if (!o->batch_event) CTOF_CUDA_TRY(cudaEventCreateWithFlags(&o->batch_event, cudaEventDisableTiming));
    CTOF_TRY(admm_graph(o, prm, st));  // made (and autotuned) before anything of this batch runs
  }
  cudaEvent_t start = ctof_ops(ks[0])->batch_event;
  CTOF_CUDA_TRY(cudaEventRecord(start, st));
  for (int i = 0; i < count; ++i) CTOF_CUDA_TRY(cudaStreamWaitEvent(ctof_ops(ks[i])->batch_stream, start, 0));
  ctof_status s = CTOF_OK;
  for (int i = 0; i < count; ++i) {
    ctof_kernel_s* o = ctof_ops(ks[i]);
    cudaStream_t side = o->batch_stream;
    if (s == CTOF_OK) s = stage_measurement(o, d_m[i], o->d_mstage, side);
    if (s == CTOF_OK && cudaGraphLaunch(o->graph, side) != cudaSuccess) s = CTOF_ECUDA;
    const size_t vb = (size_t)o->nz * o->n * o->n * sizeof(float);
    if (s == CTOF_OK && cudaMemcpyAsync(d_mu[i], o->d_vstage, vb, cudaMemcpyDeviceToDevice, side) != cudaSuccess)
      s = CTOF_ECUDA;
    // `st` waits for what was enqueued, also after an error
    if (cudaEventRecord(o->batch_event, side) != cudaSuccess ||
        cudaStreamWaitEvent(st, o->batch_event, 0) != cudaSuccess)
      s = CTOF_ECUDA;
  }
  return s;
}

}  // namespace

extern "C" {

const char* ctof_status_string(ctof_status s) {
  switch (s) {
    case CTOF_OK: return "ok";
    case CTOF_EINVAL: return "invalid argument";
    case CTOF_ENOMEM: return "out of device memory";
    case CTOF_ECUDA: return "CUDA runtime error";
    case CTOF_ENONFINITE: return "non-finite value";
    case CTOF_ETIMEOUT: return "device wait timed out";
    case CTOF_EUNSUPPORTED: return "unsupported configuration";
  }
  return "unknown status";
}

const char* ctof_last_error_message(void) { return g_last_error; }

void ctof_kernel_destroy(ctof_kernel k) {
  if (!k) return;
  DeviceGuard guard(k->device);
  for (ctof_kernel_s* o : {k->tz, k}) {  // what either operator made on first use
    if (!o) continue;
    if (o->graph) cudaGraphExecDestroy(o->graph);
    if (o->batch_stream) cudaStreamDestroy(o->batch_stream);
    if (o->batch_event) cudaEventDestroy(o->batch_event);
    destroy_events(o);
  }
  if (k->d_bt_cinv) cudaFree(k->d_bt_cinv);
  if (k->d_batch) cudaFree(k->d_batch);
  for (int i = 0; i < 2; ++i)
    if (k->d_tik_hinv[i]) cudaFree(k->d_tik_hinv[i]);
  time_basis_free(k);
  if (k->d_admm) cudaFree(k->d_admm);
  if (k->d_w) cudaFree(k->d_w);
  if (k->d_base) cudaFree(k->d_base);
  delete k;
}

namespace {

// The x-update's copies of the tables, for the operator that ADMM runs on.
ctof_status admm_copies(ctof_kernel_s* k, cudaStream_t st) {
  if (!k->tz) {
    const bool warp = contract_warp_floats(k->nt, k->nz, 0) > 0;
    Carver cv;
    const size_t o_wp = cv.take<float>(k->nclass * contract_warp_floats(k->nt, k->nz, 0));
    const size_t o_w = cv.take<float>(
        k->nclass * (warp ? contract_warp_floats(k->nt, k->nz, 1) : contract_admm_pipe_floats(k->nt, k->nz, 0)));
    const size_t o_h = cv.take<float>(
        k->nclass * (warp ? contract_warp_floats(k->nt, k->nz, 2) : contract_admm_pipe_floats(k->nt, k->nz, 1)));
    if (cv.off > 0) {
      k->admm_bytes = cv.off;
      if (cudaMalloc(&k->d_admm, k->admm_bytes) != cudaSuccess) {
        cudaGetLastError();
        k->d_admm = nullptr;
        k->admm_bytes = 0;
        return CTOF_OK;  // no room: the kernels that read d_what and d_hinv themselves
      }
      char* b = static_cast<char*>(k->d_admm);
      (warp ? k->d_what_block : k->d_what_admm) = reinterpret_cast<float*>(b + o_w);
      (warp ? k->d_hinv_block : k->d_hinv_admm) = reinterpret_cast<float*>(b + o_h);
      if (warp) k->d_what_pitch = reinterpret_cast<float*>(b + o_wp);
    }
  }
  CTOF_TRY(contract_admm_prepare(ctof_ops(k), st));
  CTOF_TRY(contract_warp_prepare(ctof_ops(k), st));
  CTOF_CUDA_TRY(cudaStreamSynchronize(st));
  return CTOF_OK;
}

ctof_status build_any(const ctof_optics* optics, const ctof_emission* emission, const ctof_voxel_average* average,
                      const ctof_grid* grid, int flags, void* stream, ctof_kernel* out) {
  if (!out) return CTOF_EINVAL;
  *out = nullptr;
  CTOF_TRY(validate(optics, grid));
  if (emission && !(isfinite(emission->mua_mm) && emission->mua_mm >= 0.0 && finite_pos(emission->musp_mm) &&
                    isfinite(emission->tau_ps) && emission->tau_ps >= 0.0))
    return CTOF_EINVAL;
  if (average) {
    if (average->layers < 0 || average->layers > grid->nz || average->nodes < 1 || average->nodes > 8)
      return CTOF_EINVAL;
    if (average->layers > 0 && grid->z_first_mm < 0.5 * grid->dz_mm) return CTOF_EINVAL;
  }
  if (flags & ~CTOF_KEEP_W) return CTOF_EINVAL;
  int dev = 0;
  CTOF_CUDA_TRY(cudaGetDevice(&dev));
  ctof_kernel_s* k = new (std::nothrow) ctof_kernel_s();
  if (!k) return CTOF_ENOMEM;
  k->optics = *optics;
  k->grid = *grid;
  k->flags = flags;
  k->fluorescence = emission ? 1 : 0;
  if (emission) k->emission = *emission;
  k->avg.layers = average ? average->layers : 0;
  k->avg.nodes = average ? average->nodes : 1;
  k->device = dev;
  k->n = grid->nx;
  k->nt = grid->nt;
  k->nz = grid->nz;
  k->p = grid->conv_mode == CTOF_LINEAR ? std::max(32, next_pow2(2 * grid->nx)) : grid->nx;
  k->h = k->p / 2 + 1;
  k->hp = ctof_round_up(k->h, 4);
  k->nf = k->p * k->h;
  k->q = grid->conv_mode == CTOF_LINEAR ? grid->nx : k->p / 2 + 1;
  k->z4 = ctof_round_up(k->nz, 4);
  k->ldt = ctof_round_up(k->nt, 8);
  k->ldz = ctof_round_up(k->nz, 8);
  k->symmetric = grid->dx_mm == grid->dy_mm;
  k->r_min = optics->clamp_r ? 0.5 * std::min(grid->dx_mm, std::min(grid->dy_mm, grid->dz_mm)) : 0.0;
  k->tik_lambda[0] = k->tik_lambda[1] = -1.0;
  k->tik_last = 1;
  k->max_polls = CTOF_DEFAULT_MAX_POLLS;
  for (int i = 0; i < 4; ++i) k->tune_pb[i] = 116;  // untuned: see tile_of in fft.cu

  std::vector<int> members;
  std::vector<float> lap;
  make_classes(k->p, k->symmetric != 0, members, lap);
  k->nclass = (int)lap.size();

  const int nt = k->nt, nz = k->nz, n = k->n, P = k->p;
  const size_t pp = (size_t)P * P;
  Carver cv;
  const size_t o_members = cv.take<int>((size_t)k->nclass * 4);
  const size_t o_lap = cv.take<float>(k->nclass);
  const size_t o_what = cv.take<float>((size_t)k->nclass * nt * k->z4);
  const size_t o_gram = cv.take<double>((size_t)k->nclass * nz * nz);
  const size_t o_hinv = cv.take<float>((size_t)k->nclass * nz * k->z4);
  const size_t o_tw = cv.take<float2>(fft_twiddle_count(P));
  const size_t o_st = cv.take<float2>((size_t)k->nf * k->ldt);
  const size_t o_st2 = cv.take<float2>((size_t)k->nf * k->ldt);
  const size_t o_sz = cv.take<float2>((size_t)k->nf * k->ldz);
  const size_t o_sz2 = cv.take<float2>((size_t)k->nf * k->ldz);
  const size_t o_it = cv.take<float2>(fft_inter_elems(k, nt, n));
  const size_t o_iz = cv.take<float2>(fft_inter_elems(k, nz, P));
  const size_t o_u1 = cv.take<float>((size_t)nt * n * n);
  const size_t o_ms = cv.take<float>((size_t)nt * n * n);
  const size_t o_u2a = cv.take<float>(3 * nz * pp);
  const size_t o_u2b = cv.take<float>(3 * nz * pp);
  const size_t o_u3 = cv.take<float>(nz * pp);
  const size_t o_xs = cv.take<float>(nz * pp);
  const size_t o_s = cv.take<float>(nz * pp);
  const size_t o_vs = cv.take<float>((size_t)nz * n * n);
  const size_t o_sc = cv.take<double>(16);
  const size_t o_fl = cv.take<int>(4);
  k->bytes = cv.off;
  if (cudaMalloc(&k->d_base, k->bytes) != cudaSuccess) {
    cudaGetLastError();
    delete k;
    return CTOF_ENOMEM;
  }
  char* b = static_cast<char*>(k->d_base);
  k->d_members = reinterpret_cast<int*>(b + o_members);
  k->d_lap = reinterpret_cast<float*>(b + o_lap);
  k->d_what = reinterpret_cast<float*>(b + o_what);
  k->d_gram = reinterpret_cast<double*>(b + o_gram);
  k->d_hinv = reinterpret_cast<float*>(b + o_hinv);
  k->d_tw = reinterpret_cast<float2*>(b + o_tw);
  k->d_spec_t = reinterpret_cast<float2*>(b + o_st);
  k->d_spec_t2 = reinterpret_cast<float2*>(b + o_st2);
  k->d_spec_z = reinterpret_cast<float2*>(b + o_sz);
  k->d_spec_z2 = reinterpret_cast<float2*>(b + o_sz2);
  k->d_inter_t = reinterpret_cast<float2*>(b + o_it);
  k->d_inter_z = reinterpret_cast<float2*>(b + o_iz);
  k->d_u1 = reinterpret_cast<float*>(b + o_u1);
  k->d_mstage = reinterpret_cast<float*>(b + o_ms);
  k->d_u2a = reinterpret_cast<float*>(b + o_u2a);
  k->d_u2b = reinterpret_cast<float*>(b + o_u2b);
  k->d_u3 = reinterpret_cast<float*>(b + o_u3);
  k->d_xs = reinterpret_cast<float*>(b + o_xs);
  k->d_s = reinterpret_cast<float*>(b + o_s);
  k->d_vstage = reinterpret_cast<float*>(b + o_vs);
  k->d_scalars = reinterpret_cast<double*>(b + o_sc);
  k->d_flags = reinterpret_cast<int*>(b + o_fl);
  if (flags & CTOF_KEEP_W) {
    void* p = nullptr;
    if (cudaMalloc(&p, (size_t)nt * nz * k->q * k->q * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      ctof_kernel_destroy(k);
      return CTOF_ENOMEM;
    }
    k->d_w = static_cast<double*>(p);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::vector<float2> tw(fft_twiddle_count(P));
  fft_twiddle_table(P, tw.data());
  ctof_status s = CTOF_OK;
  do {
    if (cudaMemsetAsync(k->d_scalars, 0, 16 * sizeof(double), st) != cudaSuccess ||
        cudaMemsetAsync(k->d_flags, 0, 4 * sizeof(int), st) != cudaSuccess ||
        cudaMemcpyAsync(k->d_members, members.data(), members.size() * sizeof(int), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(k->d_lap, lap.data(), lap.size() * sizeof(float), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(k->d_tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      s = CTOF_ECUDA;
      break;
    }
    s = build_kernel_tables(k, st);
    if (s == CTOF_OK) s = admm_copies(k, st);
  } while (0);
  if (s != CTOF_OK) {
    cudaStreamSynchronize(st);
    ctof_kernel_destroy(k);
    return s;
  }
  *out = k;
  return CTOF_OK;
}

}  // namespace

ctof_status ctof_build_kernel(const ctof_optics* optics, const ctof_grid* grid, int flags, void* stream,
                              ctof_kernel* out) {
  return build_any(optics, nullptr, nullptr, grid, flags, stream, out);
}

ctof_status ctof_build_kernel_ex(const ctof_optics* optics, const ctof_emission* emission,
                                 const ctof_voxel_average* average, const ctof_grid* grid, int flags, void* stream,
                                 ctof_kernel* out) {
  return build_any(optics, emission, average, grid, flags, stream, out);
}

ctof_status ctof_build_kernel_fluorescence(const ctof_optics* excitation, const ctof_emission* emission,
                                           const ctof_grid* grid, int flags, void* stream, ctof_kernel* out) {
  if (!emission) {
    if (out) *out = nullptr;
    return CTOF_EINVAL;
  }
  return build_any(excitation, emission, nullptr, grid, flags, stream, out);
}

ctof_status ctof_kernel_get_info(ctof_kernel k, ctof_kernel_info* info) {
  if (!k || !info) return CTOF_EINVAL;
  info->p = k->p;
  info->n_freq = k->nf;
  info->n_class = k->nclass;
  info->nt = k->nt;
  info->nz = k->nz;
  info->scale = k->scale;
  info->gram_max_diag = k->gram_max;
  const ctof_kernel_s* o = ctof_ops(k);
  info->admm_stages = o->d_what_pitch  ? contract_warp_slots(o->nt, o->nz)
                      : o->d_what_admm ? contract_admm_pipe_stages(o->nt, o->nz)
                                       : 0;
  const size_t tik_bytes = (size_t)k->nclass * k->nz * k->z4 * sizeof(float);
  info->device_bytes = k->bytes + k->admm_bytes + (k->tz ? k->tz->tz_bytes : 0) +
                       (k->d_w ? (size_t)k->nt * k->nz * k->q * k->q * sizeof(double) : 0) +
                       ((k->d_tik_hinv[0] ? 1 : 0) + (k->d_tik_hinv[1] ? 1 : 0)) * tik_bytes + k->bt_bytes +
                       k->batch_bytes;
  return CTOF_OK;
}

ctof_status ctof_kernel_get_planes(ctof_kernel k, int* planes) {
  if (!k || !planes) return CTOF_EINVAL;
  *planes = ctof_ops(k)->nt;
  return CTOF_OK;
}

const char* ctof_kernel_admm_kernel(ctof_kernel k) {
  if (!k) return "";
  const ctof_kernel_s* o = ctof_ops(k);
  return o->d_what_pitch ? "k_contract_warp" : o->d_what_admm ? "k_contract_admm_pipe" : "k_contract_admm";
}

ctof_status ctof_kernel_get_w(ctof_kernel k, double* h_w) {
  if (!k || !h_w) return CTOF_EINVAL;
  if (!k->d_w) return CTOF_EUNSUPPORTED;
  DeviceGuard g(k->device);
  CTOF_CUDA_TRY(cudaMemcpy(h_w, k->d_w, (size_t)k->nt * k->nz * k->q * k->q * sizeof(double), cudaMemcpyDeviceToHost));
  return CTOF_OK;
}

ctof_status ctof_kernel_get_classes(ctof_kernel k, int* h_members) {
  if (!k || !h_members) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  CTOF_CUDA_TRY(cudaMemcpy(h_members, k->d_members, (size_t)k->nclass * 4 * sizeof(int), cudaMemcpyDeviceToHost));
  return CTOF_OK;
}

ctof_status ctof_kernel_get_what(ctof_kernel k, float* h_what) {
  if (!k || !h_what) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  CTOF_CUDA_TRY(cudaMemcpy2D(h_what, (size_t)k->nz * sizeof(float), k->d_what, (size_t)k->z4 * sizeof(float),
                             (size_t)k->nz * sizeof(float), (size_t)k->nclass * k->nt, cudaMemcpyDeviceToHost));
  return CTOF_OK;
}

ctof_status ctof_forward(ctof_kernel k, const float* d_mu, float* d_m, void* stream) {
  if (!k || !d_mu || !d_m) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  return forward_bins(k, d_mu, d_m, false, static_cast<cudaStream_t>(stream));
}

ctof_status ctof_adjoint(ctof_kernel k, const float* d_m, float* d_vol, void* stream) {
  if (!k || !d_m || !d_vol) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ctof_kernel_s* o = ctof_ops_once(k);
  if (!o->tz_nt) return adjoint_impl(k, d_m, d_vol, st);
  CTOF_TRY(time_compress(o, 1, d_m, o->d_u1, st));
  return adjoint_impl(o, o->d_u1, d_vol, st);
}

ctof_status ctof_contract_forward_batch(ctof_kernel k, int nvol, const float* d_in, float* d_out, void* stream) {
  if (!k || !d_in || !d_out || nvol < 1) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  return contract_forward_batch(k, nvol, reinterpret_cast<const float2*>(d_in), reinterpret_cast<float2*>(d_out),
                                static_cast<cudaStream_t>(stream));
}

ctof_status ctof_contract_adjoint_batch(ctof_kernel k, int nvol, const float* d_in, float* d_out, void* stream) {
  if (!k || !d_in || !d_out || nvol < 1) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  return contract_adjoint_batch(k, nvol, reinterpret_cast<const float2*>(d_in), reinterpret_cast<float2*>(d_out),
                                static_cast<cudaStream_t>(stream));
}

ctof_status ctof_forward_multiplexed(ctof_kernel k, const float* d_mu, float* d_y, void* stream) {
  if (!k || !d_mu || !d_y) return CTOF_EINVAL;
  if (k->n % 8 != 0) return CTOF_EUNSUPPORTED;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  return forward_bins(k, d_mu, d_y, true, static_cast<cudaStream_t>(stream));
}

ctof_status ctof_adjoint_multiplexed(ctof_kernel k, const float* d_y, float* d_vol, void* stream) {
  if (!k || !d_y || !d_vol) return CTOF_EINVAL;
  if (k->n % 8 != 0) return CTOF_EUNSUPPORTED;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ctof_kernel_s* o = ctof_ops_once(k);
  CTOF_TRY(stage_measurement(o, d_y, o->d_u1, st));
  CTOF_TRY(block_hadamard(o->d_u1, o->nt, o->n, st));
  return adjoint_impl(o, o->d_u1, d_vol, st);
}

ctof_status ctof_reconstruct(ctof_kernel k, const float* d_m, const ctof_solver_params* params, float* d_mu,
                             ctof_report* report, void* stream) {
  if (!k || !d_m || !d_mu) return CTOF_EINVAL;
  CTOF_TRY(validate_params(params));
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t vbytes = (size_t)k->nz * k->n * k->n * sizeof(float);
  double lambda = 0.0;
  ctof_kernel_s* o = solver_ops(k, params);
  CTOF_TRY(stage_measurement(o, d_m, o->d_mstage, st));
  CTOF_TRY(solve_staged(o, params, &lambda, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(d_mu, k->d_vstage, vbytes, cudaMemcpyDeviceToDevice, st));
  if (report) return fill_report(k, params, lambda, report, st);
  return CTOF_OK;
}

ctof_status ctof_reconstruct_host(ctof_kernel k, const float* h_m, const ctof_solver_params* params, float* h_mu,
                                  ctof_report* report, void* stream) {
  if (!k || !h_m || !h_mu) return CTOF_EINVAL;
  CTOF_TRY(validate_params(params));
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t mbytes = (size_t)k->nt * k->n * k->n * sizeof(float);
  const size_t vbytes = (size_t)k->nz * k->n * k->n * sizeof(float);
  double lambda = 0.0;
  CTOF_CUDA_TRY(cudaMemcpyAsync(k->d_mstage, h_m, mbytes, cudaMemcpyHostToDevice, st));
  ctof_kernel_s* o = solver_ops(k, params);
  if (o->tz_nt) CTOF_TRY(time_compress(o, 1, k->d_mstage, o->d_mstage, st));
  CTOF_TRY(solve_staged(o, params, &lambda, st));
  CTOF_CUDA_TRY(cudaMemcpyAsync(h_mu, k->d_vstage, vbytes, cudaMemcpyDeviceToHost, st));
  if (report) return fill_report(k, params, lambda, report, st);
  return take_device_status(k, st);
}

ctof_status ctof_reconstruct_batch_tikhonov(ctof_kernel k, int batch, const float* d_m, int precision,
                                            int refine_steps, double lambda_rel, float* d_mu, double* lambda_out,
                                            void* stream) {
  if (!k || !d_m || !d_mu || batch < 1 || batch > 4096) return CTOF_EINVAL;
  if (refine_steps < 0 || refine_steps > 8 || !finite_pos(lambda_rel)) return CTOF_EINVAL;
  if (precision != CTOF_FP32 && precision != CTOF_BF16 && precision != CTOF_FP8E4M3) return CTOF_EINVAL;
  if (precision != CTOF_FP32 && batch_tikhonov_smem_bytes(k->nt, k->nz) > 227 * 1024) return CTOF_EUNSUPPORTED;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const double lambda = lambda_rel * k->gram_max;
  if (lambda_out) *lambda_out = lambda;
  const size_t mvol = (size_t)k->nt * k->n * k->n, xvol = (size_t)k->nz * k->n * k->n;
  if (precision == CTOF_FP32) {
    // the plain FP32 path, one volume at a time (comparison baseline)
    ctof_solver_params prm{};
    prm.solver = CTOF_SOLVER_TIKHONOV;
    prm.tik_lambda_rel = lambda_rel;
    ctof_kernel_s* o = ctof_ops_once(k);
    for (int b = 0; b < batch; ++b) {
      double lam = 0.0;
      CTOF_TRY(stage_measurement(o, d_m + b * mvol, o->d_mstage, st));
      CTOF_TRY(tikhonov_run(o, &prm, st, &lam));
      CTOF_CUDA_TRY(cudaMemcpyAsync(d_mu + b * xvol, k->d_vstage, xvol * sizeof(float), cudaMemcpyDeviceToDevice, st));
    }
    return CTOF_OK;
  }
  // FP8 keeps the time bins.  Its terms share one scale per class (W_hat) and right-hand side (m_hat), which a
  // plane that gathers a window of bins sets for all the others, and rounding errors average out over fewer
  // planes: with few depths that shows (64-bit error 1.3e-4 on the bins, 1.9e-4 on the planes at 74^2 x 3 x 368).
  const bool tz = k->tz != nullptr && precision != CTOF_FP8E4M3;
  ctof_kernel_s* own = k;
  if (tz) k = k->tz;
  const int ldm = ctof_round_up(batch * k->nt, 8), ldx = ctof_round_up(batch * k->nz, 8);
  const size_t b_sm = (size_t)k->nf * ldm * sizeof(float2), b_sx = (size_t)k->nf * ldx * sizeof(float2);
  // (the row passes pitch their planes to a multiple of 16)
  const size_t b_in = fft_inter_elems(k, batch * std::max(k->nt, k->nz), k->n) * sizeof(float2);
  const size_t b_fft = ((b_sm + 255) & ~(size_t)255) + ((b_sx + 255) & ~(size_t)255) + ((b_in + 255) & ~(size_t)255);
  const size_t need = b_fft + (tz ? (size_t)batch * k->nt * k->n * k->n * sizeof(float) : 0);
  if (need > own->batch_bytes) {
    CTOF_CUDA_TRY(cudaStreamSynchronize(st));
    if (own->d_batch) cudaFree(own->d_batch);
    own->d_batch = nullptr;
    own->batch_bytes = 0;
    if (cudaMalloc(&own->d_batch, need) != cudaSuccess) {
      cudaGetLastError();
      own->d_batch = nullptr;
      return CTOF_ENOMEM;
    }
    own->batch_bytes = need;
  }
  char* base = static_cast<char*>(own->d_batch);
  float2* spec_m = reinterpret_cast<float2*>(base);
  float2* spec_x = reinterpret_cast<float2*>(base + ((b_sm + 255) & ~(size_t)255));
  float2* inter = reinterpret_cast<float2*>(base + ((b_sm + 255) & ~(size_t)255) + ((b_sx + 255) & ~(size_t)255));
  if (tz) {
    float* planes = reinterpret_cast<float*>(base + b_fft);
    CTOF_TRY(time_compress(k, batch, d_m, planes, st));
    d_m = planes;
  }
  CTOF_TRY(fft_forward_planes(k, d_m, batch * k->nt, k->n, k->n, k->n, inter, spec_m, ldm, st));
  CTOF_TRY(batch_tikhonov_prepare(own, lambda, st));
  CTOF_TRY(batch_tikhonov_contract(k, precision, batch, spec_m, ldm, spec_x, ldx, refine_steps, st));
  return fft_inverse_planes(k, spec_x, ldx, batch * k->nz, k->n, k->n, inter, d_mu, k->n, st);
}

ctof_status ctof_kernel_autotune(ctof_kernel k, void* stream) {
  if (!k) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  for (ctof_kernel_s* o : {k, k->tz}) {
    if (!o) continue;
    o->tuned = 0;
    CTOF_TRY(autotune(o, static_cast<cudaStream_t>(stream)));
  }
  return CTOF_OK;
}

ctof_status ctof_kernel_get_tuning(ctof_kernel k, int* h_pb4) {
  if (!k || !h_pb4) return CTOF_EINVAL;
  k = ctof_ops(k);
  for (int i = 0; i < 4; ++i) h_pb4[i] = k->tune_pb[i];
  return k->tuned ? CTOF_OK : CTOF_EUNSUPPORTED;
}

ctof_status ctof_reconstruct_batch(int count, const ctof_kernel* ks, const float* const* d_m,
                                   const ctof_solver_params* params, float* const* d_mu, void* stream) {
  if (count < 1 || count > 4096 || !ks || !d_m || !d_mu) return CTOF_EINVAL;
  CTOF_TRY(validate_params(params));
  if (params->solver != CTOF_SOLVER_ADMM_TV) return CTOF_EINVAL;
  for (int i = 0; i < count; ++i) {
    if (!ks[i] || !d_m[i] || !d_mu[i] || ks[i]->device != ks[0]->device) return CTOF_EINVAL;
    for (int j = 0; j < i; ++j)
      if (ks[j] == ks[i]) return CTOF_EINVAL;  // a handle's workspace serves one problem at a time
  }
  DeviceGuard g(ks[0]->device);
  if (!g.ok) return CTOF_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return batch_run(count, ks, d_m, params, d_mu, st);
}

ctof_status ctof_set_wait_limit(ctof_kernel k, long long polls) {
  if (!k || polls < 0) return CTOF_EINVAL;
  k->max_polls = polls;
  if (k->tz) k->tz->max_polls = polls;
  return CTOF_OK;
}

ctof_status ctof_sync_status(ctof_kernel k, void* stream) {
  if (!k) return CTOF_EINVAL;
  DeviceGuard g(k->device);
  if (!g.ok) return CTOF_ECUDA;
  return take_device_status(k, static_cast<cudaStream_t>(stream));
}

ctof_status ctof_set_timing(ctof_kernel k, int enable) {
  if (!k || (enable != 0 && enable != 1)) return CTOF_EINVAL;
  ctof_ops(k)->timing = enable;
  return CTOF_OK;
}

ctof_status ctof_get_timing(ctof_kernel k, ctof_timing* out) {
  if (!k || !out) return CTOF_EINVAL;
  memset(out, 0, sizeof(*out));
  k = ctof_ops(k);
  out->graph_kernel_nodes = k->graph_kernel_nodes;
  if (!k->graph || !k->graph_timing) return CTOF_EUNSUPPORTED;
  DeviceGuard g(k->device);
  const int iters = k->graph_iters;
  CTOF_CUDA_TRY(cudaEventSynchronize(k->events[4 * iters - 1]));
  for (int it = 0; it < iters; ++it) {
    float a = 0.f, b = 0.f, c = 0.f;
    CTOF_CUDA_TRY(cudaEventElapsedTime(&a, k->events[4 * it + 0], k->events[4 * it + 1]));
    CTOF_CUDA_TRY(cudaEventElapsedTime(&b, k->events[4 * it + 1], k->events[4 * it + 2]));
    CTOF_CUDA_TRY(cudaEventElapsedTime(&c, k->events[4 * it + 2], k->events[4 * it + 3]));
    out->contract_ms += a;
    out->t_side_ms += b;
    out->z_side_ms += c;
  }
  float tot = 0.f;
  CTOF_CUDA_TRY(cudaEventElapsedTime(&tot, k->events[0], k->events[4 * iters - 1]));
  out->iterations_ms = tot;
  out->contract_launches = iters;
  return CTOF_OK;
}

}  // extern "C"
