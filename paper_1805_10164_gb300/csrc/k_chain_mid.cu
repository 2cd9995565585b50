// Block-column propagation of the RGF for 32 < W < 64 slices in FP32 (Sec. III.B), one CTA per
// pair of block columns and direction: G_{k,m} = -t g^L_k G_{k+1,m} towards slice 0 and
// G_{k,m} = -t g^R_k G_{k-1,m} towards slice L - 1, each block emitted as the Step 6' weights
// eta_{k,a} |G_{k,m}[a][b]|^2 of the column's W rows and, at the boundary slices, the lead weights
// sum_nu Gamma_nu |(Phi^T G_{k,m})_{nu b}|^2.  The same operations in the same order as
// chain_kernel (k_rgf.cu), each rounding written out, so the weights have the same bits.
//
// What bounds it: the FP32 pipe, at six operations per complex multiply-add (the product is
// rounded before it is added), the widths padded to multiples of 16 rows and columns.  A warp
// per column, as chain_kernel has it, re-reads both factors from shared memory for every
// output; here 256 threads hold the pair's W x 2W outputs, up to 4 x 8 each, so that a
// multiply-add costs a quarter of a shared-memory load.  X is overwritten in place between two
// barriers a step; the next g block is fetched into registers during the product.  Odd row
// pitches keep rows and columns free of bank conflicts.  Measured (GB300), diagonal blocks and
// columns: W=40 x L=50, 16 tasks 7.3 -> 1.15 ms; W=48 x L=50 11.4 -> 1.70; W=63 x L=40 23.2 -> 2.7.
#include <cuda_runtime.h>
#include <math.h>

#include "negf_internal.cuh"

namespace negf {
namespace {

constexpr int kMidThreads = 256;

__host__ __device__ inline size_t mid_smem_bytes(int W) {
  // X [W][2W | 1], then g [W][W | 1]
  return sizeof(cf) * ((size_t)W * ((2 * W) | 1) + (size_t)W * (W | 1));
}

// RI x CJ outputs a thread: rows ty + 16 i, columns tx + 16 j
template <int RI, int CJ>
__device__ __forceinline__ void chain_mid_body(const TaskDesc& d, const TcJob& job,
                                               const float* __restrict__ eta32,
                                               const float* __restrict__ phi32,
                                               const double* __restrict__ gam,
                                               const cf* __restrict__ gL,
                                               const cf* __restrict__ gR,
                                               const cf* __restrict__ start,
                                               float* __restrict__ weights, unsigned char* smem) {
  const int W = d.W, L = d.L, n = d.n, K = d.K, N = 2 * W, WW = W * W;
  const int XP = N | 1, GP = W | 1;
  const int tid = threadIdx.x, dir = job.dir;
  const int ty = tid >> 4, tx = tid & 15;
  cf* X = reinterpret_cast<cf*>(smem);                     // [c][b']
  cf* Gs = X + W * XP;                                     // [a][c]
  const int ys[2] = {job.y0, job.y1};
  auto m0_of = [&](int y) { return y < L ? y : (y == L ? 0 : L - 1); };
  auto row_of = [&](int y, int b) -> uint64_t {
    return y < L ? (uint64_t)y * W + b : (uint64_t)n + (uint64_t)(y - L) * W + b;
  };
  const float mt = (float)(-d.t);
  const float* eta = eta32 + d.onsite_off / 2;
  const cf* gsrc = (dir == 0 ? gL : gR) + d.g_off;
  float* wt = weights + d.wt_off;
  // (quotient, remainder) by W of tid, tid + 256, ... step by step
  const int qs = kMidThreads / W, rs = kMidThreads - qs * W;
  const int q0 = tid / W, r0 = tid - q0 * W;
  auto load_start = [&](int col) {
    const cf* st = start + d.start_off + (uint64_t)ys[col] * WW;
    for (int i = tid, c = q0, b = r0; i < WW; i += kMidThreads) {
      X[c * XP + col * W + b] = st[i];
      c += qs;
      b += rs;
      if (b >= W) { b -= W; ++c; }
    }
  };
  auto emit = [&](int k, unsigned mask) {
    for (int i = tid, r = q0, a = r0; i < N * W; i += kMidThreads) {
      const int col = r >= W;
      if (mask & (1u << col)) {
        const cf v = X[a * XP + r];
        wt[row_of(ys[col], r - col * W) * K + (uint64_t)k * W + a] =
            __fmul_rn(__ldg(eta + k * W + a), __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)));
      }
      r += qs;
      a += rs;
      if (a >= W) { a -= W; ++r; }
    }
  };
  // lead weights at a boundary slice: |(Phi^T X)_{nu b'}|^2 of every (nu, b') into the g buffer,
  // which no product needs any more (or yet), then summed over nu in order.  Synchronised before
  // and after.
  auto lead_weights = [&](int k, unsigned mask) {
    float* z2 = reinterpret_cast<float*>(Gs);              // [nu][b']
    const float* phi = phi32 + d.phi_off;
    for (int i = tid; i < N * W; i += kMidThreads) {
      const int nu = i / N, r = i - nu * N;
      float zr = 0.f, zi = 0.f;
#pragma unroll 4
      for (int a = 0; a < W; ++a) {
        const float p = __ldg(phi + a * W + nu);
        const cf v = X[a * XP + r];
        zr = __fmaf_rn(p, v.x, zr);
        zi = __fmaf_rn(p, v.y, zi);
      }
      z2[i] = __fmaf_rn(zr, zr, __fmul_rn(zi, zi));
    }
    __syncthreads();
    if (tid < N && (mask & (1u << (tid >= W)))) {
      const int col = tid >= W;
      float sum = 0.f;
      for (int nu = 0; nu < W; ++nu) sum = __fmaf_rn((float)gam[d.lead_off + nu], z2[nu * N + tid], sum);
      const uint64_t at = row_of(ys[col], tid - col * W) * K + n;
      if (k == 0) wt[at] = sum;
      if (k == L - 1) wt[at + 1] = sum;
    }
    __syncthreads();
  };
  unsigned have = 0;
  for (int col = 0; col < 2; ++col)
    if (ys[col] >= 0) have |= 1u << col;
  if (dir == 0) {
    // the start blocks themselves
    for (int col = 0; col < 2; ++col) {
      if (!(have & (1u << col))) continue;
      const int m0 = m0_of(ys[col]);
      load_start(col);
      __syncthreads();
      emit(m0, 1u << col);
      if (m0 == 0 || m0 == L - 1) lead_weights(m0, 1u << col);
    }
    __syncthreads();
  }
  const int m0a = m0_of(job.y0), m0b = job.y1 >= 0 ? m0_of(job.y1) : m0a;
  const int k_first = dir == 0 ? max(m0a, m0b) - 1 : min(m0a, m0b) + 1;
  const int k_end = dir == 0 ? -1 : L;
  const int kstep = dir == 0 ? -1 : 1;
  constexpr int kPre = RI * RI;                            // W <= 16 RI: W^2 / 256 <= RI^2
  cf gp[kPre];
  auto fetch = [&](int k) {
    const cf* gk = gsrc + (uint64_t)k * WW;
#pragma unroll
    for (int q = 0; q < kPre; ++q) {
      const int i = tid + kMidThreads * q;
      if (i < WW) gp[q] = gk[i];
    }
  };
  auto put = [&]() {
    int a = q0, c = r0;
#pragma unroll
    for (int q = 0; q < kPre; ++q) {
      if (tid + kMidThreads * q < WW) Gs[a * GP + c] = gp[q];
      a += qs;
      c += rs;
      if (c >= W) { c -= W; ++a; }
    }
  };
  if (k_first == k_end) return;
  fetch(k_first);
  put();
  // operand rows and columns; those beyond the block read its last ones and are not stored
  int ra[RI], cb[CJ];
#pragma unroll
  for (int i = 0; i < RI; ++i) ra[i] = min(ty + 16 * i, W - 1) * GP;
#pragma unroll
  for (int j = 0; j < CJ; ++j) cb[j] = min(tx + 16 * j, N - 1);
  for (int k = k_first; k != k_end; k += kstep) {
    unsigned active = 0, join = 0;
    for (int col = 0; col < 2; ++col) {
      if (!(have & (1u << col))) continue;
      const int m0 = m0_of(ys[col]);
      if (dir == 0 ? k < m0 : k > m0) active |= 1u << col;
      if (dir == 0 ? k == m0 - 1 : k == m0 + 1) join |= 1u << col;
    }
    if (join) {
      if (join & 1u) load_start(0);
      if (join & 2u) load_start(1);
      __syncthreads();                                     // (also the first g block)
    }
    const bool more = k + kstep != k_end;
    if (more) fetch(k + kstep);
    float accr[RI][CJ], acci[RI][CJ];
#pragma unroll
    for (int i = 0; i < RI; ++i)
#pragma unroll
      for (int j = 0; j < CJ; ++j) accr[i][j] = acci[i][j] = 0.f;
    for (int c = 0; c < W; ++c) {
      cf g[RI], x[CJ];
#pragma unroll
      for (int i = 0; i < RI; ++i) g[i] = Gs[ra[i] + c];
#pragma unroll
      for (int j = 0; j < CJ; ++j) x[j] = X[c * XP + cb[j]];
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < CJ; ++j) {
          accr[i][j] = __fadd_rn(accr[i][j],
                                 __fmaf_rn(g[i].x, x[j].x, -__fmul_rn(g[i].y, x[j].y)));
          acci[i][j] = __fadd_rn(acci[i][j],
                                 __fmaf_rn(g[i].y, x[j].x, __fmul_rn(g[i].x, x[j].y)));
        }
    }
    __syncthreads();                                       // X and g have been read
#pragma unroll
    for (int i = 0; i < RI; ++i)
#pragma unroll
      for (int j = 0; j < CJ; ++j) {
        const int a = ty + 16 * i, b = tx + 16 * j;
        if (a < W && b < N)
          X[a * XP + b] = cf{__fmul_rn(mt, accr[i][j]), __fmul_rn(mt, acci[i][j])};
      }
    if (more) put();
    __syncthreads();
    emit(k, active);
    if (k == 0 || k == L - 1) lead_weights(k, active);     // the last step of its direction
  }
}

__global__ void __launch_bounds__(kMidThreads, 2) chain_mid_kernel(
    const TaskDesc* __restrict__ tasks, const TcJob* __restrict__ jobs,
    const float* __restrict__ eta32, const float* __restrict__ phi32,
    const double* __restrict__ gam, const cf* __restrict__ gL, const cf* __restrict__ gR,
    const cf* __restrict__ start, float* __restrict__ weights) {
  extern __shared__ __align__(16) unsigned char smem[];
  const TcJob job = jobs[blockIdx.x];
  const TaskDesc d = tasks[job.task];
  if (d.W <= 40)
    chain_mid_body<3, 5>(d, job, eta32, phi32, gam, gL, gR, start, weights, smem);
  else if (d.W <= 48)
    chain_mid_body<3, 6>(d, job, eta32, phi32, gam, gL, gR, start, weights, smem);
  else if (d.W <= 56)
    chain_mid_body<4, 7>(d, job, eta32, phi32, gam, gL, gR, start, weights, smem);
  else
    chain_mid_body<4, 8>(d, job, eta32, phi32, gam, gL, gR, start, weights, smem);
}

}  // namespace

cudaError_t launch_chain_mid(const TaskDesc* d_tasks, const TcJob* d_jobs, uint32_t n_jobs,
                             const float* d_eta32, const float* d_phi32, const double* d_gam,
                             const void* d_gL, const void* d_gR, const void* d_start,
                             void* d_weights, cudaStream_t s) {
  if (n_jobs == 0) return cudaSuccess;
  const size_t smem = mid_smem_bytes(63);      // 94 KB: two CTAs an SM, as many as registers allow
  const cudaError_t e = allow_smem(chain_mid_kernel);
  if (e != cudaSuccess) return e;
  chain_mid_kernel<<<n_jobs, kMidThreads, smem, s>>>(
      d_tasks, d_jobs, d_eta32, d_phi32, d_gam, static_cast<const cf*>(d_gL),
      static_cast<const cf*>(d_gR), static_cast<const cf*>(d_start),
      static_cast<float*>(d_weights));
  return cudaGetLastError();
}

}  // namespace negf
