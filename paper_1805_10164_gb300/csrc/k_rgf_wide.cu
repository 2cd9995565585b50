// RGF sweeps and diagonal blocks of complex64 wires wider than 16 sites (Sec. III.B), one CTA
// per sweep or diagonal block, the W x W inversions by gj_blocked.cuh: panels on slices where
// every site dephases, partial pivoting on the others.
#include <cuda_runtime.h>
#include <math.h>

#include "gj_blocked.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

// FP32 slice block -h, staged once (multi-orbital slices), behind the shared inversion state
__host__ __device__ constexpr size_t wide_smem_bytes(bool slice_h) {
  return sizeof(BgShared) + (slice_h ? sizeof(float) * 64 * 64 : 0);
}

// Off-diagonal part of E - H_kk - Sigma_s, the same on every slice
__device__ __forceinline__ float wide_offdiag(int i, int j, float tf, const float* hs) {
  if (hs) return hs[i * 64 + j];
  return (i - j == 1 || j - i == 1) ? tf : 0.f;
}

// diagonal entry (a, a) of E - H_kk - Sigma_s of slice k, as slice_entry forms it
__device__ __forceinline__ cf wide_diag(const TaskDesc& d, const double* onsite,
                                        const double* eta, const double* h, int k, int a) {
  const double e = d.E - onsite[k * d.W + a];
  return cf{(float)(h ? e - h[a * d.W + a] : e), (float)(0.5 * eta[k * d.W + a])};
}

// One sweep (task, direction) per CTA.  A slice costs one barrier per panel of four pivots and
// one for forming its matrix, which happens while the previous slice's g is stored: the column
// warps form columns >= 4 and the panel warp, from its own registers, the first panel, which
// it then eliminates.  The next slice's diagonal is fetched by the two warps without columns.
// Measured (GB300) against one pivot at a time with 1024 threads: W=64 x L=100, 8 energies 6.81 ->
// 2.41 ms, W=64 x L=1000 66.7 -> 24.0 ms (24 us a slice); W=32 x L=100, 32 energies 1.83 -> 0.73 ms.
template <int NH>
__global__ void __launch_bounds__(kBgThreads<NH>) rgf_sweep_wide_kernel(
    const TaskDesc* __restrict__ tasks, int n_tasks, const double* __restrict__ wire, cf* gL,
    cf* gR, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int job = blockIdx.x;
  if (job >= 2 * n_tasks) return;
  const TaskDesc d = tasks[job >> 1];
  const int dir = job & 1;
  const int W = d.W, L = d.L, WW = W * W;
  if (L < 2 || W <= 16 || (NH == 1 ? W > 32 : W <= 32 || W > 64)) return;
  BgShared& S = *reinterpret_cast<BgShared*>(smem_raw);
  const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const int unit = bg_unit<NH>(warp);
  const int j = NH == 2 ? (unit & 1) * 32 + lane : lane;
  const int g = NH == 2 ? unit >> 1 : unit;
  const int NP = (W + 3) >> 2;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + d.n;
  const double* h = slice_block(d, onsite);
  float* hs = h ? reinterpret_cast<float*>(smem_raw + sizeof(BgShared)) : nullptr;
  if (h)
    for (int idx = tid; idx < WW; idx += nth) {
      const int a = idx / W, b = idx - a * W;
      hs[a * 64 + b] = 0.f - (float)h[idx];
    }
  // the slices' diagonals, one slice ahead, by the warps without columns
  const int dw = bg_side<NH>(warp);
  auto fetch_diag = [&](int s) {
    if (dw < 0 || s >= L - 1) return;
    const int a = 32 * dw + lane, k = dir == 0 ? s : L - 1 - s;
    const bool und = a < W && !(eta[k * W + a] > 0.0);
    if (a < W) S.diag[s & 1][a] = wide_diag(d, onsite, eta, h, k, a);
    const bool any = __any_sync(0xffffffffu, und);
    if (lane == 0) S.undephased[s & 1][dw] = any;
  };
  fetch_diag(0);
  if (tid == 0) S.bad = 0;
  __syncthreads();
  const cf* lb = gL + d.g_off + (uint64_t)(L - 1) * WW;   // the lead block (launch_lead_blocks)
  cf* out = (dir == 0 ? gL : gR) + d.g_off;
  const float tf = (float)d.t, tt = (float)(d.t * d.t);
  cf* Bg = S.B[NP & 1];                                   // g of the previous slice
  bool bad = false;
  // entry (i, j) of slice s: E - H - Sigma_s - (lead block, or t^2 g of the slice before, which
  // is stored on the way)
  auto form = [&](int s, int i, int c, cf* gdst) {
    const cf e = i == c ? S.diag[s & 1][i] : cf{wide_offdiag(i, c, tf, hs), 0.f};
    if (s == 0) return e - lb[i * W + c];
    const cf v = Bg[i * kBgPitch + c];
    gdst[i * W + c] = v;
    bad |= !finite_c(v);
    return cf{__fmaf_rn(-tt, v.x, e.x), __fmaf_rn(-tt, v.y, e.y)};
  };
  cf v[4], f[4], inv[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = f[c] = inv[c] = cf{0.f, 0.f};
  for (int s = 0; s < L - 1; ++s) {
    cf* gdst = s > 0 ? out + (uint64_t)(dir == 0 ? s - 1 : L - s) * WW : nullptr;
    // (expected, so that the pivoted code is laid out behind the panels': 2.46 -> 2.41 ms at W=64 x
    // L=100, 8 energies)
    if (__builtin_expect(!(S.undephased[s & 1][0] || (NH == 2 && S.undephased[s & 1][1])), 1)) {
      if (warp < NH) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (tid < W) v[c] = form(s, tid, c, gdst);
        bg_factor<NH, true>(S, 0, 4, 0, S.B[1], v, f, inv);
      } else if (unit >= 0 && j >= 4 && j < W) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int i = g + kBgGroups * r;
          if (i < W) S.B[0][i * kBgPitch + j] = form(s, i, j, gdst);
        }
      }
      __syncthreads();
      bg_invert<NH>(S, W, v, f, inv, [&] { fetch_diag(s + 1); });
    } else {
      // a site without dephasing: partial pivoting on the block in shared memory
      cf* A = bg_pivoted_in(S, W);
      for (int idx = tid; idx < WW; idx += nth) {
        const int i = idx / W, c = idx - i * W;
        A[i * kBgPitch + c] = form(s, i, c, gdst);
      }
      fetch_diag(s + 1);
      __syncthreads();
      if (!bg_pivoted(S, W)) {
        if (tid == 0) atomicOr(err, ERR_SINGULAR);
        return;
      }
    }
  }
  cf* gdst = out + (uint64_t)(dir == 0 ? L - 2 : 1) * WW;
  for (int idx = tid; idx < WW; idx += nth) {
    const int i = idx / W, c = idx - i * W;
    const cf x = Bg[i * kBgPitch + c];
    gdst[idx] = x;
    bad |= !finite_c(x);
  }
  if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERR_NONFINITE);
  if (tid == 0 && S.bad) atomicOr(err, ERR_SINGULAR);
}

// last task whose first job index is <= job
__device__ __forceinline__ int wide_task(const TaskDesc* tasks, int n_tasks, uint32_t job) {
  int lo = 0, hi = n_tasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].col_base <= job) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Diagonal blocks: one CTA per (task, y) as diag_cta_kernel (k_rgf.cu), same outputs.  Two CTAs an SM
// at W <= 32: with one (106 registers) batches of short narrow wires were slower than by that
// kernel (W=17 x L=20, 64 energies 0.063 ms there, 0.090 with one, 0.062 with two; W=32 x L=100, 32
// energies 0.246, 0.240, 0.164).
template <int NH>
__global__ void __launch_bounds__(kBgThreads<NH>, NH == 1 ? 2 : 1) diag_wide_kernel(
    const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t n_jobs,
    const double* __restrict__ wire, const double* __restrict__ phig,
    const double* __restrict__ gam, const cf* __restrict__ gL, const cf* __restrict__ gR,
    cf* __restrict__ start, double* __restrict__ rowsum, double* __restrict__ mode_w,
    double* __restrict__ cvals, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t job = blockIdx.x;
  if (job >= n_jobs) return;
  const int task = wide_task(tasks, n_tasks, job);
  const TaskDesc d = tasks[task];
  const int W = d.W, L = d.L, n = d.n, WW = W * W;
  if (W <= 16 || (NH == 1 ? W > 32 : W <= 32 || W > 64)) return;
  BgShared& S = *reinterpret_cast<BgShared*>(smem_raw);
  const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const int unit = bg_unit<NH>(warp);
  const int j = NH == 2 ? (unit & 1) * 32 + lane : lane;
  const int g = NH == 2 ? unit >> 1 : unit;
  const int NP = (W + 3) >> 2;
  const int y = (int)(job - d.col_base);
  const bool inj = y >= L;
  const int p = y - L;
  const int m0 = inj ? (p == 0 ? 0 : L - 1) : y;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + n;
  const double* h = slice_block(d, onsite);
  const double* phi = phig + d.phi_off;
  const float tf = (float)d.t, tt = (float)(d.t * d.t);
  const bool lead_l = m0 == 0, lead_r = m0 == L - 1;
  const cf* lb = gL + d.g_off + (uint64_t)(L - 1) * WW;   // the lead block
  const cf* gl = gL + d.g_off + (uint64_t)(lead_l ? 0 : m0 - 1) * WW;
  const cf* gr = gR + d.g_off + (uint64_t)(lead_r ? 0 : m0 + 1) * WW;
  // E - H - Sigma_s - (lead block or t^2 g^L_{m-1}) - (lead block or t^2 g^R_{m+1})
  auto form = [&](int i, int c) {
    cf e = i == c ? S.diag[0][i]
                  : cf{h ? 0.f - (float)h[i * W + c] : wide_offdiag(i, c, tf, nullptr), 0.f};
    const int idx = i * W + c;
    const cf l = lead_l ? lb[idx] : cf{__fmul_rn(tt, gl[idx].x), __fmul_rn(tt, gl[idx].y)};
    const cf r = lead_r ? lb[idx] : cf{__fmul_rn(tt, gr[idx].x), __fmul_rn(tt, gr[idx].y)};
    return cf{__fsub_rn(__fsub_rn(e.x, l.x), r.x), __fsub_rn(__fsub_rn(e.y, l.y), r.y)};
  };
  if (tid < W) S.diag[0][tid] = wide_diag(d, onsite, eta, h, m0, tid);
  if (tid == 0) S.bad = 0;
  const bool deph = __syncthreads_and(tid >= W || eta[m0 * W + tid] > 0.0);
  cf* G = S.B[NP & 1];
  cf* T = S.B[(NP & 1) ^ 1];                              // free once the inverse is in G
  if (deph) {
    cf v[4], f[4], inv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[c] = inv[c] = cf{0.f, 0.f};
    if (warp < NH) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (tid < W) v[c] = form(tid, c);
      bg_factor<NH, true>(S, 0, 4, 0, S.B[1], v, f, inv);
    } else if (unit >= 0 && j >= 4 && j < W) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int i = g + kBgGroups * r;
        if (i < W) S.B[0][i * kBgPitch + j] = form(i, j);
      }
    }
    __syncthreads();
    bg_invert<NH>(S, W, v, f, inv, [] {});
    if (S.bad) {
      if (tid == 0) atomicOr(err, ERR_SINGULAR);
      return;
    }
  } else {
    cf* A = bg_pivoted_in(S, W);
    for (int idx = tid; idx < WW; idx += nth) {
      const int i = idx / W, c = idx - i * W;
      A[i * kBgPitch + c] = form(i, c);
    }
    __syncthreads();
    if (!bg_pivoted(S, W)) {
      if (tid == 0) atomicOr(err, ERR_SINGULAR);
      return;
    }
  }
  // start block: G_mm, or G_mm Phi for the injection columns
  cf* dst = start + d.start_off + (uint64_t)y * WW;
  const cf* R = inj ? T : G;
  bool bad = false;
  for (int idx = tid; idx < WW; idx += nth) {
    const int a = idx / W, b = idx - a * W;
    cf v;
    if (!inj) {
      v = G[a * kBgPitch + b];
    } else {
      v = cf{0.f, 0.f};
      for (int c = 0; c < W; ++c) v = v + (float)phi[c * W + b] * G[a * kBgPitch + c];
      T[a * kBgPitch + b] = v;
    }
    dst[idx] = v;
    bad |= !finite_c(v);
  }
  if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERR_NONFINITE);
  // A per row: site b: -2 Im G_bb;  mode mu: -2 Im (Phi^T G Phi)_{mu mu}
  double* mw_s = reinterpret_cast<double*>(S.F);
  for (int b = tid; b < W; b += nth) {
    if (!inj) {
      rowsum[d.row_base + m0 * W + b] = -2.0 * (double)R[b * kBgPitch + b].y;
    } else {
      double im = 0.0;
      for (int a = 0; a < W; ++a) im += phi[a * W + b] * (double)R[a * kBgPitch + b].y;
      const double Ab = -2.0 * im;
      rowsum[d.row_base + n + p * W + b] = Ab;
      const double mw = gam[d.lead_off + b] * Ab;
      mode_w[d.mode_off + p * W + b] = mw;
      mw_s[b] = mw;
    }
  }
  __syncthreads();
  if (inj && tid == 0) {
    double c = 0.0;
    for (int b = 0; b < W; ++b) c += mw_s[b];      // fixed order
    cvals[task * 2 + p] = c;
    rowsum[d.row_base + d.rows + p] = c;
  }
}

}  // namespace

cudaError_t launch_rgf_sweep_wide(const TaskDesc* d_tasks, int n_tasks, int max_W,
                                  const double* d_wire, cf* d_gL, cf* d_gR, int32_t* d_err,
                                  cudaStream_t s) {
  // widths 17 .. 32 and 33 .. 64 by kernels of their own; each skips the other's tasks
  const size_t smem = wide_smem_bytes(true);
  cudaError_t e = allow_smem(rgf_sweep_wide_kernel<1>);
  if (e == cudaSuccess) e = allow_smem(rgf_sweep_wide_kernel<2>);
  if (e != cudaSuccess) return e;
  if (max_W > 32) {
    rgf_sweep_wide_kernel<2><<<2 * n_tasks, kBgThreads<2>, smem, s>>>(d_tasks, n_tasks, d_wire,
                                                                     d_gL, d_gR, d_err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  rgf_sweep_wide_kernel<1><<<2 * n_tasks, kBgThreads<1>, smem, s>>>(d_tasks, n_tasks, d_wire,
                                                                   d_gL, d_gR, d_err);
  return cudaGetLastError();
}

cudaError_t launch_diag_wide(const TaskDesc* d_tasks, int n_tasks, uint32_t n_cols, int max_W,
                             const double* d_wire, const double* d_phi, const double* d_gam,
                             const cf* d_gL, const cf* d_gR, cf* d_start, double* d_rowsum,
                             double* d_mode_w, double* d_c, int32_t* d_err, cudaStream_t s) {
  const size_t smem = wide_smem_bytes(false);
  cudaError_t e = allow_smem(diag_wide_kernel<1>);
  if (e == cudaSuccess) e = allow_smem(diag_wide_kernel<2>);
  if (e != cudaSuccess) return e;
  if (max_W > 32) {
    diag_wide_kernel<2><<<n_cols, kBgThreads<2>, smem, s>>>(d_tasks, n_tasks, n_cols, d_wire,
                                                            d_phi, d_gam, d_gL, d_gR, d_start,
                                                            d_rowsum, d_mode_w, d_c, d_err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  diag_wide_kernel<1><<<n_cols, kBgThreads<1>, smem, s>>>(d_tasks, n_tasks, n_cols, d_wire, d_phi,
                                                          d_gam, d_gL, d_gR, d_start, d_rowsum,
                                                          d_mode_w, d_c, d_err);
  return cudaGetLastError();
}

}  // namespace negf
