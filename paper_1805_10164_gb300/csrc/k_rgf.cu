// Lead self-energies, RGF sweeps and the block-column / transition-weight kernels.
//
// Sec. III.B: the paper obtains G^r by the recursive Green's function algorithm (RGF), the
// diagonal once per sample and one column of G^r per walker step.  Here every column a table
// row needs is produced once per (wire, energy) task:
//   * lead_modes_kernel   - eigen self-energies Sigma_m and Gamma_m of the lead strips
//                           (Sec. II.A lead self-energies; Sec. III.A model)
//   * lead_block_kernel   - Phi diag(Sigma_m) Phi^T, the leads' self-energy on the sites
//   * rgf_sweep_*_kernel  - left- and right-connected blocks g^L_k, g^R_k (one warp per task
//                           and direction in registers for complex64 W <= 16, one CTA
//                           otherwise, k_rgf_wide.cu for complex64; the sweep is a serial chain
//                           of W x W inversions)
//   * diag_*_kernel       - per slice m: G_mm by one more inversion; for the boundary slices
//                           also G Phi, the A of every row (for the sum-rule check), the mode
//                           weights of Eq. lead_out_probability and c_p = Tr[Gamma_p A]
//                           (Eq. elast_lin_xpq)
//   * chain_*_kernel      - per slice m and direction, the block column
//                           G_{k,m} = -t g^L_k G_{k+1,m} (k < m), -t g^R_k G_{k-1,m} (k > m),
//                           emitted directly as Step 6' weights (Eq. draw_i_simult and the lead
//                           probability of Step 6'); the two injection columns propagate G Phi
//                           for the rows of Steps 4-5.
// W x W block inversions are Gauss-Jordan: in registers by one warp for complex64 W <= 16, by
// one CTA otherwise (gj.cuh, gj_blocked.cuh); partial pivoting except on slices where every site
// dephases (see gj_rows).  All of it runs in the precision of the tables: complex128 for
// NEGF_FP64, complex64 for NEGF_FP32; the lead self-energies, whose square roots are singular
// at the sub-band edges, are FP64 in both and rounded once.
#include <cuda_runtime.h>
#include <math.h>

#include "gj.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

// Sine mode phi_m(a) of a W-site cross-section, m, a in [0, W).
__device__ __forceinline__ double phi_mode(int a, int m, int W) {
  return sqrt(2.0 / (W + 1)) * sinpi((double)((m + 1) * (a + 1)) / (double)(W + 1));
}

__global__ void lead_modes_kernel(const TaskDesc* __restrict__ tasks, int n_tasks,
                                  const double* __restrict__ wire, double* phi, float* phi32,
                                  float* eta32, cd* sig, double* gam, int32_t* err) {
  const int task = blockIdx.x;
  if (task >= n_tasks) return;
  const TaskDesc d = tasks[task];
  if (d.e_idx == 0) {
    // once per wire: transverse modes (a multi-orbital slice's come from slice_modes_kernel)
    // and the FP32 copy of eta
    if (!d.slice_h)
      for (int idx = threadIdx.x; idx < d.W * d.W; idx += blockDim.x) {
        const double v = phi_mode(idx / d.W, idx % d.W, d.W);
        phi[d.phi_off + idx] = v;
        phi32[d.phi_off + idx] = (float)v;
      }
    const double* eta = wire + d.onsite_off + d.n;
    for (int i = threadIdx.x; i < d.n; i += blockDim.x) eta32[d.onsite_off / 2 + i] = (float)eta[i];
  }
  for (int m = threadIdx.x; m < d.W; m += blockDim.x) {
    cd s;
    double g;
    if (d.lead_model == NEGF_LEAD_WIDE_BAND) {
      s = mk(0.0, -0.5 * d.gamma_lead);
      g = d.gamma_lead;
    } else {
      // eps_m = -2t cos((m+1) pi / (W+1)) (a slice block: its m-th eigenvalue);
      // Sigma_m = t^2 g_s(E - eps_m), retarded branch
      const double eps = d.slice_h
                             ? wire[d.onsite_off + 2 * (uint64_t)d.n + (uint64_t)d.W * d.W + m]
                             : -2.0 * d.t * cospi((double)(m + 1) / (double)(d.W + 1));
      const double e = d.E - eps, two_t = 2.0 * d.t;
      if (fabs(fabs(e) - two_t) <= 1e-12 * d.t) atomicOr(err, ERR_INPUT);
      if (fabs(e) < two_t) {
        const double r = sqrt(two_t * two_t - e * e);
        s = mk(0.5 * e, -0.5 * r);
        g = r;
      } else {
        const double r = sqrt(e * e - two_t * two_t);
        s = mk(0.5 * (e - copysign(r, e)), 0.0);
        g = 0.0;
      }
    }
    sig[d.lead_off + m] = s;
    gam[d.lead_off + m] = g;
  }
}

// The lead block Phi diag(sigma) Phi^T of every task (both leads alike), summed in FP64 and
// rounded to the blocks' precision, into the last slice's slot of g^L (the left-connected block
// of slice L - 1 is never needed).  One thread per entry a >= b, mirrored.  The sum takes W
// dependent FP64 steps per entry; formed inside every sweep and boundary diagonal block, one
// CTA at a time on the narrow FP64 pipe, it cost 0.2 ms of latency per kernel at W = 64.
// Wires of up to kOwnLeadW sites form it within the register sweeps (complex64), which saves the
// smallest builds a launch: W=1 x L=1 0.099 -> 0.093 ms.
constexpr int kLeadBlockThreads = 64;
constexpr int kOwnLeadW = 4;

// entry (a, b) of Phi diag(sigma) Phi^T
__device__ __forceinline__ cd lead_entry(int a, int b, int W, const double* phi, const cd* sg) {
  cd acc = mk(0.0, 0.0);
  for (int m = 0; m < W; ++m) acc = acc + (phi[a * W + m] * phi[b * W + m]) * sg[m];
  return acc;
}

template <typename C>
__global__ void __launch_bounds__(kLeadBlockThreads) lead_block_kernel(
    const TaskDesc* __restrict__ tasks, int chunks, const double* __restrict__ phig,
    const cd* __restrict__ sig, C* __restrict__ gL) {
  const TaskDesc& d = tasks[blockIdx.x / chunks];
  const int W = d.W;
  const int e = (blockIdx.x % chunks) * kLeadBlockThreads + threadIdx.x;
  if (e >= W * (W + 1) / 2) return;
  int a = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while (a * (a + 1) / 2 > e) --a;
  while ((a + 1) * (a + 2) / 2 <= e) ++a;
  const int b = e - a * (a + 1) / 2;
  const cd acc = lead_entry(a, b, W, phig + d.phi_off, sig + d.lead_off);
  C* lb = gL + d.g_off + (uint64_t)(d.L - 1) * W * W;
  lb[a * W + b] = lb[b * W + a] = to_c(acc, C{});
}

// ---- CTA-wide complex128 inversions (any W <= 64) ------------------------------------------
// cta_gj (gj.cuh): the slice block sits in shared memory and is inverted in place by
// Gauss-Jordan (no augmented identity):
//   pivot k:  a_kk <- 1/a_kk;  a_kj <- a_kj / a_kk;  a_ik <- -a_ik / a_kk;
//             a_ij <- a_ij - (a_ik / a_kk) a_kj            (i, j != k)
// with two barriers per pivot: the pivot row (1/a_kk formed once, in a_kk's slot) and the
// pivot column are copied out, then every thread updates its entries with a_kj / a_kk formed
// once per thread.  Thread t owns column t mod W of rows t / W, t / W + R,
// ... (R = threads / W), so that a warp touches consecutive entries of one row.  On a
// slice where every site dephases no pivot search is needed (see gj_rows); otherwise rows are
// interchanged by partial pivoting and the inverse's columns unscrambled at the end.  The
// diagonal blocks use it, and every sweep on slices with an undephased site.
//
// The sweeps (rgf_sweep_rows_kernel) keep the block in registers instead: thread t owns column
// j = t mod W of rows g, g + RG, g + 2 RG, ...
// (g = t / W, RG = ceil(W / RPT) row groups of at most RPT rows), and a pivot costs one
// barrier: the owners of row k publish it and the owners of column k publish that column, into
// one of two buffers (alternating with k, so that the next pivot's writes cannot overtake this
// pivot's reads); then every warp forms 1/a_kk for itself, its even lanes dividing for the real
// part and its odd lanes for the imaginary part, and every thread updates its rows.  What
// bounds a pivot is the chain of FP64 instructions of its busiest warp, since a warp's FP64
// instruction holds its scheduler's share of the pipe for 64 cycles, so RPT is the smallest for
// which kSweepRowsThreads threads hold the block: a W = 10 block takes four warps with one row a
// thread.  Measured, GB300, W=10 x L=50, 64 energies: 1.55 -> 0.54 ms against four rows a thread
// (one warp) and the reciprocal formed by a_kk's owner; W=24 x L=40 4.48 -> 2.01; W=64 x L=30
// 22.0 -> 15.5.  The next slice's matrix E - H - Sigma_s - t^2 g_k is formed in the same
// registers while g_k is stored.
constexpr int kSweepThreads = 256;       // diagonal blocks: many CTAs
constexpr int kSweepRowsThreads = 256;   // complex128 sweeps
constexpr int kSweepRegMaxW = 16;        // complex64 sweeps up to this width: one warp each

template <typename C>
__host__ __device__ inline size_t sweep_rows_bytes(int W) {
  // A W x W | pivot rows 2 x 64 | pivot columns 2 x 64 (complex) | perm 64, flag (int)
  return sizeof(C) * (size_t)(W * W + 4 * 64) + sizeof(int) * (size_t)(64 + 2);
}

// In-place inverse of the register-held block (see above; no pivot search: the caller takes
// it on slices where every site dephases, gj_rows says why that is safe).  i_m = g + RG m are
// this thread's rows, valid while i_m < W; false (uniformly) on a zero or non-finite pivot.
template <typename C, int RPT>
__device__ bool gj_regcols(C (&a)[RPT], int W, int RG, int g, int j, bool own, C* rowk,
                           C* fcol) {
  using R = typename Real<C>::T;
  const bool odd = threadIdx.x & 1;
  const bool warp_owns = (int)(threadIdx.x & ~31u) < RG * W;
  bool bad = false;
  int kr = 0, km = 0;                       // pivot k = kr + RG km: its row group and slot
  for (int k = 0; k < W; ++k) {
    const int b = k & 1;
    C* rk = rowk + 64 * b;
    C* fc = fcol + 64 * b;
    if (own && g == kr) {
      C v = a[0];
#pragma unroll
      for (int m = 1; m < RPT; ++m)
        if (m == km) v = a[m];
      rk[j] = v;
    }
    if (own && j == k) {
#pragma unroll
      for (int m = 0; m < RPT; ++m)
        if (g + RG * m < W) fc[g + RG * m] = a[m];
    }
    __syncthreads();
    if (warp_owns) {
      // 1/a_kk: the even lanes divide for its real part, the odd ones for its imaginary part
      const C p = rk[k];
      const R dd = p.x * p.x + p.y * p.y;
      const R q = (odd ? (R)0 - p.y : p.x) / dd;
      const R o = __shfl_xor_sync(0xffffffffu, q, 1);
      const C inv = odd ? C{o, q} : C{q, o};
      bad |= !finite_c(inv);
      if (own) {
        // a_ij - a_ik t with t = a_kj / a_kk; column k: 0 - a_ik / a_kk.  One code path for
        // both: a branch would send the warp through the FP64 pipe twice
        const C t = j == k ? inv : rk[j] * inv;
#pragma unroll
        for (int m = 0; m < RPT; ++m) {
          const int i = g + RG * m;
          if (i < W) {
            const C v = (j == k ? mkc(0.0, 0.0, C{}) : a[m]) - fc[i] * t;
            a[m] = i == k ? t : v;
          }
        }
      }
    }
    if (++kr == RG) {
      kr = 0;
      ++km;
    }
  }
  return !__syncthreads_or(bad);
}

template <typename C, int RPT>
__device__ __forceinline__ void sweep_rows_body(const TaskDesc& d, int dir,
                                               const double* __restrict__ wire, C* gL, C* gR,
                                               int32_t* err, unsigned char* smem_raw) {
  using R = typename Real<C>::T;
  const int W = d.W, L = d.L, WW = W * W;
  const int tid = threadIdx.x;
  const int RG = (W + RPT - 1) / RPT;
  const int j = tid % W, g = tid / W;
  const bool own = g < RG;
  C* A = reinterpret_cast<C*>(smem_raw);   // the block, for the pivoted inversion only
  C* rowk = A + WW;
  C* fcol = rowk + 2 * 64;
  int* perm = reinterpret_cast<int*>(fcol + 2 * 64);
  int* flag = perm + 64;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + d.n;
  // first slice of the sweep: E - H - Sigma_s - the lead block
  const C* lb = gL + d.g_off + (uint64_t)(L - 1) * WW;
  const int kf = dir == 0 ? 0 : L - 1;
  C a[RPT];
#pragma unroll
  for (int m = 0; m < RPT; ++m) {
    const int i = g + RG * m;
    a[m] = mkc(0.0, 0.0, C{});
    if (own && i < W)
      a[m] = slice_entry<C>(i, j, kf, W, d.E, d.t, onsite, eta, slice_block(d, onsite)) -
             lb[i * W + j];
  }
  C* out = dir == 0 ? gL : gR;
  const R tt = (R)(d.t * d.t);
  for (int s = 0; s < L - 1; ++s) {
    const int k = dir == 0 ? s : L - 1 - s;
    const bool deph = __syncthreads_and(tid >= W || eta[k * W + tid] > 0.0);
    bool ok;
    if (deph) {
      ok = gj_regcols<C, RPT>(a, W, RG, g, j, own, rowk, fcol);
    } else {
      // an undephased site: partial pivoting on the block in shared memory
#pragma unroll
      for (int m = 0; m < RPT; ++m)
        if (own && g + RG * m < W) A[(g + RG * m) * W + j] = a[m];
      __syncthreads();
      ok = cta_gj(A, rowk, fcol, perm, flag, W, true);
      __syncthreads();
#pragma unroll
      for (int m = 0; m < RPT; ++m)
        if (own && g + RG * m < W) a[m] = A[(g + RG * m) * W + j];
    }
    if (!ok) {
      if (tid == 0) atomicOr(err, ERR_SINGULAR);
      return;
    }
    // store g_k; form the next slice: E - H - Sigma_s - t^2 g_k
    C* dst = out + d.g_off + (uint64_t)k * WW;
    const bool more = s + 1 < L - 1;
    const int kn = dir == 0 ? s + 1 : L - 2 - s;
    bool bad = false;
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
      const int i = g + RG * m;
      if (own && i < W) {
        const C v = a[m];
        dst[i * W + j] = v;
        bad |= !finite_c(v);
        if (more) a[m] = slice_entry<C>(i, j, kn, W, d.E, d.t, onsite, eta, slice_block(d, onsite)) - tt * v;
      }
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERR_NONFINITE);
  }
}

__global__ void __launch_bounds__(kSweepRowsThreads) rgf_sweep_rows_kernel(
    const TaskDesc* __restrict__ tasks, int n_tasks, const double* __restrict__ wire, cd* gL,
    cd* gR, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int job = blockIdx.x;
  if (job >= 2 * n_tasks) return;
  const TaskDesc d = tasks[job >> 1];
  const int dir = job & 1;
  if (d.L < 2 || d.W > 64) return;
  // rows per thread: the fewest with which kSweepRowsThreads threads hold the block
  if (d.W <= 16)
    sweep_rows_body<cd, 1>(d, dir, wire, gL, gR, err, smem_raw);
  else if (d.W <= 22)
    sweep_rows_body<cd, 2>(d, dir, wire, gL, gR, err, smem_raw);
  else if (d.W <= 32)
    sweep_rows_body<cd, 4>(d, dir, wire, gL, gR, err, smem_raw);
  else if (d.W <= 42)
    sweep_rows_body<cd, 8>(d, dir, wire, gL, gR, err, smem_raw);
  else
    sweep_rows_body<cd, 16>(d, dir, wire, gL, gR, err, smem_raw);
}

// ---- register-resident variants for complex64 blocks with W <= 16 ------------------------
// Lane i < W holds row i of the augmented matrix [M | I] in registers: a[0, MAXW) the slice
// matrix, a[MAXW, 2 MAXW) the identity (then the inverse).  Gauss-Jordan pivots without moving
// rows: at step k the pivot is the unused row with the largest |a_ik|^2 (one warp max-reduction
// of a 32-bit key), the pivot lane publishes its row in shared memory (broadcast loads cost far
// less than two shuffles per element), and every other row eliminates column k.  Row i of the inverse then sits in the lane that pivoted column i.  The kernels call
// these with MAXW equal to the block width, so that every column index is a constant.

// Gauss-Jordan on the register-held rows; on return lane i < W holds row i of the inverse in
// a[MAXW, MAXW + W).  Returns false uniformly on a zero or non-finite pivot.
//
// At step k the pivot lane computes 1 / a_pk itself and publishes it with its row as it stands;
// every other row subtracts (a_ik / a_pk) times that row.  Pivot rows are not rescaled during
// the elimination (a pivot row only ever changes by multiples of later pivot rows, so it stays
// a_pk times its normalised form); each is divided by its own pivot at the end.  This keeps the
// reciprocal off the other lanes' dependency chain.
//
// pivot == false eliminates in row order without a pivot search.  The caller takes it only when
// every site of the slice dephases (eta_i > 0): the slice matrix E - H - Sigma is then complex
// symmetric with imaginary part >= diag(eta / 2) > 0 (the lead and connected-block terms add
// positive semidefinite imaginary parts, since Im G^r <= 0), its Schur complements keep that
// property, so no pivot vanishes and elimination without pivoting is stable for this class.
// The row goes through shared memory as 16-byte pairs of entries: on a lone warp each shared
// memory (or shuffle) instruction costs about as much as a dozen arithmetic ones, so the
// broadcast is made of as few, and as wide, accesses as possible.
// srow: 2 W + 2 complex64 of this warp's shared memory, 16-byte aligned.
template <int W>
__device__ bool gj_rows(cf (&a)[2 * W], bool pivot, cf* srow) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  float4* row = reinterpret_cast<float4*>(srow);   // row[q]: entries 2q, 2q + 1; row[W]: 1/pivot
  bool used = lane >= W;                           // lanes without a row never pivot
  int src = lane;
  cf own_inv{1.f, 0.f};                            // 1 / pivot of the step this lane pivoted
#pragma unroll
  for (int k = 0; k < W; ++k) {
    int p = k;
    if (pivot) {
      // key: |a_ik|^2 (non-negative, so its bits order like the value) with its low 5 mantissa
      // bits replaced by 31 - lane: the largest candidate wins, lower lanes on near-ties
      const float v = used ? 0.f : norm2(a[k]);
      const unsigned key = (__float_as_uint(v) & ~31u) | (unsigned)(31 - lane);
      const unsigned best = __reduce_max_sync(FULL, key);
      const unsigned mag = best & ~31u;
      if (mag == 0u || mag >= 0x7f800000u) return false;   // zero, inf or NaN pivot
      p = 31 - (int)(best & 31u);
      if (lane == k) src = p;
    }
    const bool me = lane == p;
    __syncwarp();                                  // the previous step's row has been read
    if (me) {
      const float rr = __frcp_rn(norm2(a[k]));      // inf for a zero pivot: caught below
      own_inv = cf{a[k].x * rr, -a[k].y * rr};
      row[W] = make_float4(own_inv.x, own_inv.y, 0.f, 0.f);
#pragma unroll
      for (int q = (k + 1) / 2; q < W; ++q)
        row[q] = make_float4(a[2 * q].x, a[2 * q].y, a[2 * q + 1].x, a[2 * q + 1].y);
    }
    __syncwarp();
    const float4 iv = row[W];
    if (!pivot && !(isfinite(iv.x) && isfinite(iv.y) && (iv.x != 0.f || iv.y != 0.f)))
      return false;
    const cf f = me ? cf{0.f, 0.f} : a[k] * cf{iv.x, iv.y};
#pragma unroll
    for (int q = (k + 1) / 2; q < W; ++q) {
      const float4 r = row[q];
      if (2 * q > k) a[2 * q] = a[2 * q] - f * cf{r.x, r.y};
      a[2 * q + 1] = a[2 * q + 1] - f * cf{r.z, r.w};
    }
    used |= me;
  }
#pragma unroll
  for (int j = W; j < 2 * W; ++j) {
    a[j] = a[j] * own_inv;
    if (pivot) {
      a[j].x = __shfl_sync(FULL, a[j].x, src);
      a[j].y = __shfl_sync(FULL, a[j].y, src);
    }
  }
  return true;
}

// In-place Gauss-Jordan inversion without pivoting: lane j < W holds column j of the matrix in
// a[0, W) on entry and column j of its inverse on return.  At step k the pivot column is
// broadcast through shared memory and every lane updates its own column from registers:
//   lane j != k:  a_kj <- a_kj / a_kk,  a_ij <- a_ij - a_ik a_kj / a_kk  (i != k)
//   lane k:       a_kk <- 1 / a_kk,     a_ik <- -a_ik / a_kk             (i != k)
// (both written as a_ij - c_i piv with piv = a_kj / a_kk, or 1 + 1 / a_kk on lane k).  Only for
// matrices whose imaginary part is positive definite (see gj_rows).  Returns false uniformly on
// a zero or non-finite pivot.  scol: W + 1 complex64 of shared memory, 16-byte aligned.
template <int W>
__device__ bool gj_cols(cf (&a)[W], cf* scol) {
  const int lane = threadIdx.x & 31;
  float4* col = reinterpret_cast<float4*>(scol);
  constexpr int W2 = (W + 1) / 2;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    __syncwarp();                                  // the previous column has been read
    if (lane == k) {
#pragma unroll
      for (int q = 0; q < W2; ++q)
        col[q] = make_float4(a[2 * q].x, a[2 * q].y, 2 * q + 1 < W ? a[2 * q + 1].x : 0.f,
                             2 * q + 1 < W ? a[2 * q + 1].y : 0.f);
    }
    __syncwarp();
    cf c[2 * W2];
#pragma unroll
    for (int q = 0; q < W2; ++q) {
      const float4 v = col[q];
      c[2 * q] = cf{v.x, v.y};
      c[2 * q + 1] = cf{v.z, v.w};
    }
    const float m = norm2(c[k]);
    if (!(m > 0.f) || !isfinite(m)) return false;
    const float rr = __frcp_rn(m);
    const cf inv{c[k].x * rr, -c[k].y * rr};
    const bool me = lane == k;
    const cf piv = me ? cf{1.f + inv.x, inv.y} : a[k] * inv;
#pragma unroll
    for (int i = 0; i < W; ++i)
      if (i != k) a[i] = a[i] - c[i] * piv;
    a[k] = me ? inv : piv;
  }
  return true;
}

// Inverse of the W x W slice matrix A held by columns (lane j < W: column j in a).  Slices where
// every site dephases take gj_cols; the others the pivoted row routine applied to A^T (lane j's
// column of A is row j of A^T, and row j of (A^T)^-1 is column j of A^-1).  Lanes >= W must hold
// zeros.  buf: 2 W + 2 complex64 of shared memory, 16-byte aligned.
template <int W>
__device__ bool invert_slice(cf (&a)[W], bool all_dephase, cf* buf) {
  if (all_dephase) return gj_cols<W>(a, buf);
  const int lane = threadIdx.x & 31;
  cf ar[2 * W];
#pragma unroll
  for (int j = 0; j < W; ++j) {
    ar[j] = a[j];
    ar[W + j] = cf{(lane < W && lane == j) ? 1.f : 0.f, 0.f};
  }
  if (!gj_rows<W>(ar, true, buf)) return false;
#pragma unroll
  for (int j = 0; j < W; ++j) a[j] = ar[W + j];
  return true;
}

// Column j (lane j < W) of E - H_kk - Sigma_s(k) - x, where x is this lane's column; other lanes
// get zero columns.
template <int W>
__device__ void build_col(cf (&a)[W], double E, double t, double onsite_j, double eta_j,
                          const cf (&x)[W], const double* h = nullptr) {
  const int j = threadIdx.x & 31;
  if (h) {
    // multi-orbital slice block: column j of E - h - diag(onsite) + i eta / 2 - x
#pragma unroll
    for (int i = 0; i < W; ++i) {
      cf v{0.f, 0.f};
      if (j < W)
        v = cf{(float)((i == j ? E - onsite_j : 0.0) - h[i * W + j]),
               i == j ? (float)(0.5 * eta_j) : 0.f} - x[i];
      a[i] = v;
    }
    return;
  }
  const cf diag{(float)(E - onsite_j), (float)(0.5 * eta_j)};
  const float tf = (float)t;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    cf v{0.f, 0.f};
    if (j < W) {
      if (i == j) v = diag;
      if (i - j == 1 || j - i == 1) v.x += tf;
      v = v - x[i];
    }
    a[i] = v;
  }
}

// column (lane < W) of the lead block at lb; other lanes get zeros
template <int W>
__device__ __forceinline__ void lead_col(const cf* lb, cf (&x)[W]) {
  const int j = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < W; ++i) x[i] = j < W ? lb[i * W + j] : cf{0.f, 0.f};
}

// One sweep (task d, direction dir) with W == MAXW known at compile time.
template <int MAXW>
__device__ __forceinline__ void sweep_reg_body(const TaskDesc& d, int dir,
                                               const double* __restrict__ wire,
                                               const double* __restrict__ phig,
                                               const cd* __restrict__ sig, cf* gL, cf* gR,
                                               int32_t* err, cf* srow) {
  constexpr int W = MAXW;
  const int L = d.L;
  const int lane = threadIdx.x & 31;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + d.n;
  const float ttf = (float)(d.t * d.t);     // FP32 on the serial path (FP64 is slow here)
  cf x[MAXW], a[MAXW];
  cf* lb = gL + d.g_off + (uint64_t)(L - 1) * W * W;
  if (W <= kOwnLeadW) {
    // (one of the two sweeps keeps it for the diagonal blocks)
#pragma unroll
    for (int i = 0; i < W; ++i) {
      x[i] = cf{0.f, 0.f};
      if (lane < W) {
        x[i] = to_c(lead_entry(i > lane ? i : lane, i > lane ? lane : i, W, phig + d.phi_off,
                               sig + d.lead_off), cf{});
        if (dir == 0) lb[i * W + lane] = x[i];
      }
    }
  } else {
    lead_col<W>(lb, x);
  }
  cf* out = dir == 0 ? gL : gR;
  const int jc = lane < W ? lane : 0;
  // the next slice's onsite energy and dephasing are fetched one step ahead
  int k = dir == 0 ? 0 : L - 1;
  double on_j = onsite[k * W + jc], eta_j = eta[k * W + jc];
  for (int s = 0; s < L - 1; ++s) {
    k = dir == 0 ? s : L - 1 - s;
    const double on_cur = on_j, eta_cur = eta_j;
    if (s + 1 < L - 1) {
      const int kn = dir == 0 ? s + 1 : L - 2 - s;
      on_j = onsite[kn * W + jc];
      eta_j = eta[kn * W + jc];
    }
    build_col<W>(a, d.E, d.t, on_cur, eta_cur, x, slice_block(d, onsite));
    const bool deph = __all_sync(0xffffffffu, lane >= W || eta_cur > 0.0);
    if (!invert_slice<W>(a, deph, srow)) {
      if (lane == 0) atomicOr(err, ERR_SINGULAR);
      return;
    }
    // lane j holds column j of g_k: store it (rows i at i W + j, coalesced over the lanes) and
    // keep t^2 times it as the next slice's column j of x
    cf* dst = out + d.g_off + (uint64_t)k * W * W + jc;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      if (lane < W) {
        dst[(uint64_t)i * W] = a[i];
        bad |= !finite_c(a[i]);
      }
      x[i] = cf{ttf * a[i].x, ttf * a[i].y};
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(err, ERR_NONFINITE);
  }
}

// Calls Body<W>::run(args...) for the compile-time W equal to w (1 <= w <= 16).
template <template <int> class Body, typename... Args>
__device__ __forceinline__ void by_width(int w, Args&&... args) {
  switch (w) {
    case 1: Body<1>::run(args...); break;
    case 2: Body<2>::run(args...); break;
    case 3: Body<3>::run(args...); break;
    case 4: Body<4>::run(args...); break;
    case 5: Body<5>::run(args...); break;
    case 6: Body<6>::run(args...); break;
    case 7: Body<7>::run(args...); break;
    case 8: Body<8>::run(args...); break;
    case 9: Body<9>::run(args...); break;
    case 10: Body<10>::run(args...); break;
    case 11: Body<11>::run(args...); break;
    case 12: Body<12>::run(args...); break;
    case 13: Body<13>::run(args...); break;
    case 14: Body<14>::run(args...); break;
    case 15: Body<15>::run(args...); break;
    case 16: Body<16>::run(args...); break;
    default: break;
  }
}

template <int W>
struct SweepReg {
  template <typename... A>
  __device__ __forceinline__ static void run(A... a) { sweep_reg_body<W>(a...); }
};

// One warp per (task, direction), tasks of width W <= kSweepRegMaxW.
__global__ void rgf_sweep_reg_kernel(const TaskDesc* __restrict__ tasks, int n_tasks,
                                     const double* __restrict__ wire,
                                     const double* __restrict__ phig,
                                     const cd* __restrict__ sig, cf* gL, cf* gR, int32_t* err) {
  const int job = blockIdx.x;
  if (job >= 2 * n_tasks) return;
  __shared__ __align__(16) cf s_row[34];
  const TaskDesc d = tasks[job >> 1];
  if (d.L < 2 && d.W > kOwnLeadW) return;
  by_width<SweepReg>(d.W, d, job & 1, wire, phig, sig, gL, gR, err, s_row);
}

// last task whose first job index (`first(t)`) is <= job
template <typename F>
__device__ __forceinline__ int find_task(int n_tasks, uint32_t job, F first) {
  int lo = 0, hi = n_tasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first(mid) <= job) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// CTA-wide complex128 diagonal blocks: one CTA of kSweepThreads threads per (task, y); same
// outputs as diag_reg_kernel, with the inversion of cta_gj.
__host__ __device__ inline size_t diag_cta_bytes(int W) {
  // A, S (start block) W x W | pivot row, multipliers W (complex) | phi W x W double | mode
  // weights W double | perm W, flag (int)
  return sizeof(cd) * (size_t)(2 * W * W + 2 * W) + sizeof(double) * (size_t)(W * W + W) +
         sizeof(int) * (size_t)(W + 2);
}

__global__ void __launch_bounds__(kSweepThreads) diag_cta_kernel(
    const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t n_jobs,
    const double* __restrict__ wire, const double* __restrict__ phig,
    const double* __restrict__ gam, const cd* __restrict__ gL, const cd* __restrict__ gR,
    cd* __restrict__ start, double* __restrict__ rowsum, double* __restrict__ mode_w,
    double* __restrict__ cvals, int32_t* err) {
  using C = cd;
  using R = double;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t job = blockIdx.x;
  if (job >= n_jobs) return;
  const int task = find_task(n_tasks, job, [&](int t) { return tasks[t].col_base; });
  const TaskDesc d = tasks[task];
  const int W = d.W, L = d.L, n = d.n, WW = W * W;
  if (W > 64) return;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int y = (int)(job - d.col_base);
  const bool inj = y >= L;
  const int p = y - L;
  const int m0 = inj ? (p == 0 ? 0 : L - 1) : y;
  C* A = reinterpret_cast<C*>(smem_raw);
  C* S = A + WW;
  C* rowk = S + WW;
  C* fcol = rowk + W;
  double* phi = reinterpret_cast<double*>(fcol + W);
  double* mw_s = phi + WW;
  int* perm = reinterpret_cast<int*>(mw_s + W);
  int* flag = perm + W;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + n;
  const R tt = (R)(d.t * d.t);
  const bool lead_l = m0 == 0, lead_r = m0 == L - 1;
  for (int idx = tid; idx < WW; idx += nth) phi[idx] = phig[d.phi_off + idx];
  // A = E - H - Sigma_s - (lead block or t^2 g^L_{m-1}) - (lead block or t^2 g^R_{m+1})
  const C* lb = gL + d.g_off + (uint64_t)(L - 1) * WW;
  const C* gl = lead_l ? nullptr : gL + d.g_off + (uint64_t)(m0 - 1) * WW;
  const C* gr = lead_r ? nullptr : gR + d.g_off + (uint64_t)(m0 + 1) * WW;
  for (int idx = tid; idx < WW; idx += nth) {
    const int a = idx / W, b = idx - a * W;
    C v = slice_entry<C>(a, b, m0, W, d.E, d.t, onsite, eta, slice_block(d, onsite));
    v = v - (gl ? tt * gl[idx] : lb[idx]);
    v = v - (gr ? tt * gr[idx] : lb[idx]);
    A[idx] = v;
  }
  const bool deph = __syncthreads_and(tid >= W || eta[m0 * W + tid] > 0.0);
  if (!cta_gj(A, rowk, fcol, perm, flag, W, !deph)) {
    if (tid == 0) atomicOr(err, ERR_SINGULAR);
    return;
  }
  // start block: G_mm, or G_mm Phi for the injection columns
  C* dst = start + d.start_off + (uint64_t)y * WW;
  bool bad = false;
  for (int idx = tid; idx < WW; idx += nth) {
    C v;
    if (!inj) {
      v = A[idx];
    } else {
      const int a = idx / W, b = idx - a * W;
      v = mkc(0.0, 0.0, C{});
      for (int c = 0; c < W; ++c) v = v + (R)phi[c * W + b] * A[a * W + c];
    }
    S[idx] = v;
    dst[idx] = v;
    bad |= !finite_c(v);
  }
  if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERR_NONFINITE);
  // A per row: site b: -2 Im G_bb;  mode mu: -2 Im (Phi^T G Phi)_{mu mu}
  for (int b = tid; b < W; b += nth) {
    if (!inj) {
      rowsum[d.row_base + m0 * W + b] = -2.0 * (double)S[b * W + b].y;
    } else {
      double im = 0.0;
      for (int a = 0; a < W; ++a) im += phi[a * W + b] * (double)S[a * W + b].y;
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

// Register-resident diagonal-block kernel (complex64, W <= MAXW <= 16); same outputs as
// diag_kernel.  Shared memory per warp: G (W x W complex64) and phi (W x W double).
template <int MAXW>
__device__ __forceinline__ void diag_reg_body(const TaskDesc& d, int task, uint32_t job,
                                              const double* __restrict__ wire,
                                              const double* __restrict__ phig,
                                              const double* __restrict__ gam,
                                              const cf* __restrict__ gL,
                                              const cf* __restrict__ gR, cf* __restrict__ start,
                                              double* __restrict__ rowsum,
                                              double* __restrict__ mode_w,
                                              double* __restrict__ cvals, int32_t* err, cf* sG,
                                              double* phi, double* s_mw, cf* srow) {
  constexpr int W = MAXW;
  const int lane = threadIdx.x & 31;
  const int L = d.L, n = d.n;
  const int y = (int)(job - d.col_base);
  const bool inj = y >= L;
  const int p = y - L;
  const int m0 = inj ? (p == 0 ? 0 : L - 1) : y;
  const double* onsite = wire + d.onsite_off;
  const double* eta = onsite + n;
  const double tt = d.t * d.t;
  for (int idx = lane; idx < W * W; idx += 32) phi[idx] = phig[d.phi_off + idx];
  // this lane's column of left + right (lead block or t^2 g)
  cf x[MAXW], a[MAXW];
  const bool lead_l = m0 == 0, lead_r = m0 == L - 1;
  if (lead_l || lead_r) {
    lead_col<W>(gL + d.g_off + (uint64_t)(L - 1) * W * W, x);
    if (lead_l && lead_r) {
#pragma unroll
      for (int i = 0; i < MAXW; ++i) x[i] = 2.f * x[i];
    }
  } else {
#pragma unroll
    for (int i = 0; i < MAXW; ++i) x[i] = cf{0.f, 0.f};
  }
  const int jc = lane < W ? lane : 0;
  const cf* gl = lead_l ? nullptr : gL + d.g_off + (uint64_t)(m0 - 1) * W * W;
  const cf* gr = lead_r ? nullptr : gR + d.g_off + (uint64_t)(m0 + 1) * W * W;
#pragma unroll
  for (int i = 0; i < MAXW; ++i) {
    if (lane < W) {
      if (gl) x[i] = x[i] + (float)tt * gl[i * W + jc];
      if (gr) x[i] = x[i] + (float)tt * gr[i * W + jc];
    }
  }
  const double eta_j = eta[m0 * W + jc];
  build_col<W>(a, d.E, d.t, onsite[m0 * W + jc], eta_j, x, slice_block(d, onsite));
  const bool deph = __all_sync(0xffffffffu, lane >= W || eta_j > 0.0);
  if (!invert_slice<W>(a, deph, srow)) {
    if (lane == 0) atomicOr(err, ERR_SINGULAR);
    return;
  }
  bool bad = false;
#pragma unroll
  for (int i = 0; i < MAXW; ++i) {
    if (lane < W) {
      sG[i * W + lane] = a[i];
      bad |= !finite_c(a[i]);
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(err, ERR_NONFINITE);
  __syncwarp();
  // start block: G_mm, or G_mm Phi for the injection columns
  cf* dst = start + d.start_off + (uint64_t)y * W * W;
  for (int idx = lane; idx < W * W; idx += 32) {
    cf v;
    if (!inj) {
      v = sG[idx];
    } else {
      const int r = idx / W, b = idx % W;
      v = cf{0.f, 0.f};
      for (int c = 0; c < W; ++c) v = v + (float)phi[c * W + b] * sG[r * W + c];
    }
    dst[idx] = v;
  }
  // A per row: site b: -2 Im G_bb;  mode mu: -2 sum_{a,c} phi_mu(a) phi_mu(c) Im G_ac
  for (int b = lane; b < W; b += 32) {
    if (!inj) {
      rowsum[d.row_base + m0 * W + b] = -2.0 * (double)sG[b * W + b].y;
    } else {
      double im = 0.0;
      for (int r = 0; r < W; ++r) {
        double row_im = 0.0;
        for (int c = 0; c < W; ++c) row_im += phi[c * W + b] * (double)sG[r * W + c].y;
        im += phi[r * W + b] * row_im;
      }
      const double A = -2.0 * im;
      rowsum[d.row_base + n + p * W + b] = A;
      const double mw = gam[d.lead_off + b] * A;
      mode_w[d.mode_off + p * W + b] = mw;
      s_mw[b] = mw;
    }
  }
  __syncwarp();
  if (inj && lane == 0) {
    double c = 0.0;
    for (int b = 0; b < W; ++b) c += s_mw[b];            // fixed order
    cvals[task * 2 + p] = c;
    rowsum[d.row_base + d.rows + p] = c;
  }
}

template <int W>
struct DiagReg {
  template <typename... A>
  __device__ __forceinline__ static void run(A... a) { diag_reg_body<W>(a...); }
};

// Register-resident diagonal blocks (complex64, W <= 16), one warp per column job; same outputs
// as diag_cta_kernel.  Shared memory per warp: G (W x W complex64), phi (W x W double), the mode
// weights.
__global__ void diag_reg_kernel(const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t n_jobs,
                                const double* __restrict__ wire, const double* __restrict__ phig,
                                const double* __restrict__ gam, const cf* __restrict__ gL,
                                const cf* __restrict__ gR,
                                cf* __restrict__ start, double* __restrict__ rowsum,
                                double* __restrict__ mode_w, double* __restrict__ cvals,
                                int32_t* err) {
  __shared__ cf s_G[8][16 * 16];
  __shared__ double s_phi[8][16 * 16];
  __shared__ double s_mw[8][16];
  __shared__ __align__(16) cf s_row[8][34];
  const int warp = threadIdx.x >> 5;
  const uint32_t job = blockIdx.x * (blockDim.x >> 5) + warp;
  if (job >= n_jobs) return;
  const int task = find_task(n_tasks, job, [&](int t) { return tasks[t].col_base; });
  const TaskDesc d = tasks[task];
  by_width<DiagReg>(d.W, d, task, job, wire, phig, gam, gL, gR, start, rowsum, mode_w,
                    cvals, err, s_G[warp], s_phi[warp], s_mw[warp], s_row[warp]);
}

template <typename C>
__host__ __device__ inline size_t chain_warp_bytes(int W) {
  // X0, X1, Gb : W x W complex | phi : W x W real | lgam : W real
  return sizeof(C) * (size_t)(3 * W * W) + sizeof(typename Real<C>::T) * (size_t)(W * W + W);
}

// One warp per (task, y, direction): the block column of start slice m0 propagated towards
// slice 0 (direction 0, which also emits the start block) or towards slice L-1 (direction 1),
// each block emitted as Step 6' weights of the column's W rows.
template <typename C>
__global__ void chain_kernel(const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t n_jobs,
                             int max_W, const typename Real<C>::T* __restrict__ eta_all,
                             const typename Real<C>::T* __restrict__ phig,
                             const double* __restrict__ gam, const C* __restrict__ gL,
                             const C* __restrict__ gR, const C* __restrict__ start,
                             typename Real<C>::T* __restrict__ weights, C* __restrict__ green,
                             C* __restrict__ gphi) {
  using R = typename Real<C>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t job = blockIdx.x * (blockDim.x >> 5) + warp;
  if (job >= n_jobs) return;
  const int task = find_task(n_tasks, job, [&](int t) { return 2 * tasks[t].col_base; });
  const TaskDesc d = tasks[task];
  if (d.fused || d.cta_chain) return;            // emitted by the tensor-core / CTA chains
  const int W = d.W, L = d.L, n = d.n, K = d.K;
  const uint32_t local = job - 2 * d.col_base;
  const int y = (int)(local >> 1), dir = (int)(local & 1);
  const bool inj = y >= L;
  const int p = y - L;
  const int m0 = inj ? (p == 0 ? 0 : L - 1) : y;
  if (dir == 1 && m0 == L - 1) return;           // nothing towards slice L-1
  unsigned char* base = smem_raw + (size_t)warp * chain_warp_bytes<C>(max_W);
  C* X0 = reinterpret_cast<C*>(base);
  C* X1 = X0 + W * W;
  C* Gb = X1 + W * W;
  R* phi = reinterpret_cast<R*>(Gb + W * W);
  R* lgam = phi + W * W;
  // eta in the table precision: the FP64 wire array (+ n past onsite) or its FP32 copy
  const R* eta = eta_all + (sizeof(R) == 8 ? d.onsite_off + n : d.onsite_off / 2);
  const R mt = (R)(-d.t);
  for (int idx = lane; idx < W * W; idx += 32) {
    phi[idx] = phig[d.phi_off + idx];
    X0[idx] = start[d.start_off + (uint64_t)y * W * W + idx];
  }
  for (int m = lane; m < W; m += 32) lgam[m] = (R)gam[d.lead_off + m];
  __syncwarp();
  const int row0 = inj ? n + p * W : m0 * W;
  R* wrow = weights + d.wt_off;
  // weights of block k held in X (X[a][b] = G_{(k,a),(m0,b)} or (G Phi)_{(k,a),mu})
  // idx / W without an integer division: (idx + 1/2) / W is at least 1/(2W) away from an
  // integer, far above the float error for idx < W^2 <= 4096
  const float rW = 1.0f / (float)W;
  auto emit = [&](const C* X, int k) {
    for (int idx = lane; idx < W * W; idx += 32) {
      const int b = (int)(((float)idx + 0.5f) * rW), a = idx - b * W;
      wrow[(uint64_t)(row0 + b) * K + k * W + a] = eta[k * W + a] * norm2(X[a * W + b]);
      if (green) {
        // keep G (site columns) or G Phi (injection columns) for the gradient
        if (!inj) green[d.green_off + (uint64_t)(k * W + a) * n + m0 * W + b] = X[a * W + b];
        else gphi[d.gphi_off + (uint64_t)(k * W + a) * 2 * W + p * W + b] = X[a * W + b];
      }
    }
    if (k == 0 || k == L - 1) {
      // lead weight of row b: sum_nu Gamma_nu |(Phi^T X)_{nu b}|^2 = <psi_b|Gamma_lead|psi_b>
      for (int b = lane; b < W; b += 32) {
        R sum = 0;
        for (int nu = 0; nu < W; ++nu) {
          C acc = C{0, 0};
          for (int a = 0; a < W; ++a) acc = acc + phi[a * W + nu] * X[a * W + b];
          sum += lgam[nu] * norm2(acc);
        }
        if (k == 0) wrow[(uint64_t)(row0 + b) * K + n + 0] = sum;
        if (k == L - 1) wrow[(uint64_t)(row0 + b) * K + n + 1] = sum;
      }
    }
  };
  C* cur = X0;
  C* nxt = X1;
  if (dir == 0) emit(cur, m0);
  const int k_end = dir == 0 ? -1 : L;
  const int step = dir == 0 ? -1 : 1;
  const C* gsrc = dir == 0 ? gL : gR;
  // the next block g_k is loaded into registers one step ahead (lane's entries idx = lane + 32 i)
  constexpr int kPre = 4;                        // covers W * W <= 128 entries
  const bool pre = W * W <= 32 * kPre;
  C gpre[kPre];
  auto fetch = [&](int k) {
    const C* gk = gsrc + d.g_off + (uint64_t)k * W * W;
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int idx = lane + 32 * i;
      if (idx < W * W) gpre[i] = gk[idx];
    }
  };
  if (pre && m0 + step != k_end) fetch(m0 + step);
  for (int k = m0 + step; k != k_end; k += step) {
    if (pre) {
#pragma unroll
      for (int i = 0; i < kPre; ++i) {
        const int idx = lane + 32 * i;
        if (idx < W * W) Gb[idx] = gpre[i];
      }
      if (k + step != k_end) fetch(k + step);
    } else {
      const C* gk = gsrc + d.g_off + (uint64_t)k * W * W;
      for (int idx = lane; idx < W * W; idx += 32) Gb[idx] = gk[idx];
    }
    __syncwarp();
    for (int idx = lane; idx < W * W; idx += 32) {
      const int a = (int)(((float)idx + 0.5f) * rW), b = idx - a * W;
      C acc = C{0, 0};
      for (int c = 0; c < W; ++c) acc = acc + Gb[a * W + c] * cur[c * W + b];
      nxt[idx] = mt * acc;
    }
    __syncwarp();
    C* tmp = cur; cur = nxt; nxt = tmp;
    emit(cur, k);
    __syncwarp();
  }
}

// Complex128 block columns without kept G: one warp per (task, y).  G = G^T, so the chains run
// towards slice 0 only (y < L: from slice y; the injection columns of lead L from slice 0 to
// slice L-1, those of lead R back), and a step emits its block G_{k,m} twice: as the weights of
// slice m's rows and, transposed, as those of slice k's.  The injection columns pass every
// (G Phi)_k, which holds the lead weights of slice k's rows.  Bound by the FP64 pipe (two lanes a cycle
// per SM): four fused multiply-adds per complex product, and half the products of both
// directions.  A pair of consecutive warps takes a long and a short chain (y and L - 1 - y), the
// longer one first or second by the parity of the pair's bits, so that every CTA and, within an
// SM, every scheduler's share of the pipe gets about the same work; loops stay rolled (the kernel
// of a tiny call is bound by its instruction fetches).  Measured, GB300, diagonal blocks and
// columns against one warp per direction: W=10 x L=50, 64 energies 3.25 -> 1.50 ms (the columns
// alone 3.0 -> 1.24, the pipe 87 % active while an SM has work); W=16 x L=100, 16 energies
// 9.56 -> 4.29; W=24 x L=40, 4 energies 4.11 -> 3.28; W=64 x L=30, 2 energies 54.0 -> 40.8.
__global__ void __maxnreg__(80) chain_sym_kernel(const TaskDesc* __restrict__ tasks, int n_tasks,
                                 uint32_t n_jobs, int max_W, const double* __restrict__ wire,
                                 const double* __restrict__ phig, const double* __restrict__ gam,
                                 const cd* __restrict__ gL, const cd* __restrict__ gR,
                                 const cd* __restrict__ start, double* __restrict__ weights) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t job = blockIdx.x * (blockDim.x >> 5) + warp;
  if (job >= n_jobs) return;
  const int task = find_task(n_tasks, job, [&](int t) { return tasks[t].col_base; });
  const TaskDesc d = tasks[task];
  if (d.fused || d.cta_chain) return;
  const int W = d.W, L = d.L, n = d.n, K = d.K, WW = W * W;
  const int i = (int)(job - d.col_base);
  const int q = i >> 1;
  const int y = i >= L ? i : ((i ^ __popc(q)) & 1) ? L - 1 - q : q;
  const bool inj = y >= L, up = y == L;
  const int m0 = inj ? (up ? 0 : L - 1) : y;
  cd* X0 = reinterpret_cast<cd*>(smem_raw + (size_t)warp * chain_warp_bytes<cd>(max_W));
  cd* X1 = X0 + WW;
  cd* Gb = X1 + WW;
  double* phi = reinterpret_cast<double*>(Gb + WW);
  double* lgam = phi + WW;
  const double* eta = wire + d.onsite_off + n;
  for (int idx = lane; idx < WW; idx += 32) {
    phi[idx] = phig[d.phi_off + idx];
    X0[idx] = start[d.start_off + (uint64_t)y * WW + idx];
  }
  for (int m = lane; m < W; m += 32) lgam[m] = gam[d.lead_off + m];
  __syncwarp();
  double* wt = weights + d.wt_off;
  const int row0 = inj ? n + (y - L) * W : m0 * W;
  // idx / W without an integer division (see chain_kernel)
  const float rW = 1.0f / (float)W;
  auto div_w = [&](int idx) { return (int)(((float)idx + 0.5f) * rW); };
  cd* cur = X0;
  cd* nxt = X1;
  const double mt = -d.t;
  const bool split = W >= 4;
  const int k_end = up ? L : -1, step = up ? 1 : -1;
  const cd* gsrc = (up ? gR : gL) + d.g_off;
  // the next block g_k is loaded into registers one step ahead (lane's entries idx = lane + 32 i)
  constexpr int kPre = 4;                        // covers W * W <= 128 entries
  const bool pre = WW <= 32 * kPre;
  cd gpre[kPre];
#pragma unroll 1
  for (int k = m0;; k += step) {
    const int kn = k + step;
    if (pre && kn != k_end) {
      const cd* gk = gsrc + (uint64_t)kn * WW;
#pragma unroll
      for (int q = 0; q < kPre; ++q)
        if (lane + 32 * q < WW) gpre[q] = gk[lane + 32 * q];
    }
    // weights of block k (cur[a][b] = G_{(k,a),(m0,b)} or (G Phi)_{(k,a),mu}), |cur|^2 kept in sq
    double* sq = reinterpret_cast<double*>(nxt);
#pragma unroll 1
    for (int idx = lane; idx < WW; idx += 32) {
      const int b = div_w(idx), a = idx - b * W;
      const double q = norm2(cur[a * W + b]);
      wt[(uint64_t)(row0 + b) * K + k * W + a] = eta[k * W + a] * q;
      sq[idx] = q;
    }
    __syncwarp();
    if (inj) {
      // the rows of slice k: <psi_a|Gamma|psi_a> = sum_nu Gamma_nu |(G Phi)_{(k,a),nu}|^2
      for (int a = lane; a < W; a += 32) {
        double sum = 0.0;
#pragma unroll 1
        for (int nu = 0; nu < W; ++nu) sum = fma(lgam[nu], sq[nu * W + a], sum);
        wt[(uint64_t)(k * W + a) * K + n + (y - L)] = sum;
      }
      // the injection rows themselves: sum_nu Gamma_nu |(Phi^T X)_{nu b}|^2
      if (k == 0 || k == L - 1) {
        __syncwarp();
#pragma unroll 1
        for (int idx = lane; idx < WW; idx += 32) {
          const int nu = div_w(idx), b = idx - nu * W;
          double re = 0.0, im = 0.0;
#pragma unroll 1
          for (int a = 0; a < W; ++a) {
            const double f = phi[a * W + nu];
            re = fma(f, cur[a * W + b].x, re);
            im = fma(f, cur[a * W + b].y, im);
          }
          sq[idx] = norm2(cd{re, im});
        }
        __syncwarp();
        for (int b = lane; b < W; b += 32) {
          double sum = 0.0;
#pragma unroll 1
          for (int nu = 0; nu < W; ++nu) sum = fma(lgam[nu], sq[nu * W + b], sum);
          double* lw = wt + (uint64_t)(row0 + b) * K + n;
          if (k == 0) lw[0] = sum;
          if (k == L - 1) lw[1] = sum;
        }
      }
    } else if (k != m0) {
#pragma unroll 1
      for (int idx = lane; idx < WW; idx += 32) {
        const int a = div_w(idx), b = idx - a * W;
        wt[(uint64_t)(k * W + a) * K + m0 * W + b] = eta[m0 * W + b] * sq[b * W + a];
      }
    }
    if (kn == k_end) break;
    if (pre) {
#pragma unroll
      for (int q = 0; q < kPre; ++q)
        if (lane + 32 * q < WW) Gb[lane + 32 * q] = gpre[q];
    } else {
      const cd* gk = gsrc + (uint64_t)kn * WW;
      for (int idx = lane; idx < WW; idx += 32) Gb[idx] = gk[idx];
    }
    __syncwarp();
#pragma unroll 1
    for (int idx = lane; idx < WW; idx += 32) {
      const int a = div_w(idx), b = idx - a * W;
      // partial sums of the four real products, from W = 4 of even and odd c apart: a fused
      // multiply-add each, and no more rounding than one sum over c of rounded complex products
      double p[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      auto mac = [&](int c, double* o) {
        const cd u = Gb[a * W + c], v = cur[c * W + b];
        o[0] = fma(u.x, v.x, o[0]);
        o[1] = fma(u.y, v.y, o[1]);
        o[2] = fma(u.x, v.y, o[2]);
        o[3] = fma(u.y, v.x, o[3]);
      };
      int c = 0;
#pragma unroll 1
      for (; split && c + 1 < W; c += 2) {
        mac(c, p);
        mac(c + 1, p + 4);
      }
#pragma unroll 1
      for (; c < W; ++c) mac(c, p);
      if (split)
        for (int m = 0; m < 4; ++m) p[m] += p[m + 4];
      nxt[idx] = cd{mt * (p[0] - p[1]), mt * (p[2] + p[3])};
    }
    __syncwarp();
    cd* tmp = cur; cur = nxt; nxt = tmp;
  }
}

int warps_for(size_t per_warp, int max_warps) {
  int w = max_warps;
  while (w > 1 && per_warp * w > 96 * 1024) --w;
  return w;
}

// Most warps per chain CTA that fit the opt-in shared memory (and 16 warps).
template <typename C>
int chain_max(int max_W) {
  const size_t per = chain_warp_bytes<C>(max_W);
  int w = 16;
  while (w > 1 && per * w > 200 * 1024) --w;
  return w;
}

template <typename C>
cudaError_t lead_blocks(const TaskDesc* d_tasks, int n_tasks, int max_W, const double* d_phi,
                        const cd* d_sig, C* d_gL, cudaStream_t s) {
  const int chunks = (max_W * (max_W + 1) / 2 + kLeadBlockThreads - 1) / kLeadBlockThreads;
  lead_block_kernel<C><<<(unsigned)(n_tasks * chunks), kLeadBlockThreads, 0, s>>>(
      d_tasks, chunks, d_phi, d_sig, d_gL);
  return cudaGetLastError();
}

cudaError_t sweep_fp64(const TaskDesc* d_tasks, int n_tasks, int max_W, const double* d_wire,
                       cd* d_gL, cd* d_gR, int32_t* d_err, cudaStream_t s) {
  // one CTA per sweep: each sweep is a serial chain of W x W inversions, spread one per SM
  const size_t smem = sweep_rows_bytes<cd>(max_W);
  const cudaError_t e = allow_smem(rgf_sweep_rows_kernel);
  if (e != cudaSuccess) return e;
  rgf_sweep_rows_kernel<<<2 * n_tasks, kSweepRowsThreads, smem, s>>>(d_tasks, n_tasks, d_wire,
                                                                     d_gL, d_gR, d_err);
  return cudaGetLastError();
}

cudaError_t sweep_fp32(const TaskDesc* d_tasks, int n_tasks, int max_W, const double* d_wire,
                       const double* d_phi, const cd* d_sig, cf* d_gL, cf* d_gR, int32_t* d_err,
                       cudaStream_t s) {
  // one warp per sweep for the tasks of width <= 16 (it skips wider ones), a CTA per sweep for
  // the rest
  rgf_sweep_reg_kernel<<<2 * n_tasks, 32, 0, s>>>(d_tasks, n_tasks, d_wire, d_phi, d_sig, d_gL,
                                                  d_gR, d_err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || max_W <= kSweepRegMaxW) return e;
  return launch_rgf_sweep_wide(d_tasks, n_tasks, max_W, d_wire, d_gL, d_gR, d_err, s);
}

template <typename C>
cudaError_t columns_impl(const TaskDesc* d_tasks, int n_tasks, uint32_t n_cols, int max_W,
                         const double* d_wire, const typename Real<C>::T* d_eta,
                         const double* d_phi, const typename Real<C>::T* d_phiR,
                         const double* d_gam, const C* d_gL, const C* d_gR, C* d_start,
                         typename Real<C>::T* d_w, double* d_rowsum, double* d_mode_w,
                         double* d_c, int32_t* d_err, C* d_green, C* d_gphi, cudaStream_t s,
                         int chain_warps, int cols_max_W) {
  if (sizeof(C) == sizeof(cf)) {
    // register-resident diagonal blocks for the tasks of width <= 16, 4 warps per block (the
    // kernel skips wider tasks)
    const int warps = 4;
    const unsigned blocks = (n_cols + warps - 1) / warps;
    const cf* gl = reinterpret_cast<const cf*>(d_gL);
    const cf* gr = reinterpret_cast<const cf*>(d_gR);
    cf* st = reinterpret_cast<cf*>(d_start);
    diag_reg_kernel<<<blocks, 32 * warps, 0, s>>>(d_tasks, n_tasks, n_cols, d_wire, d_phi, d_gam,
                                                  gl, gr, st, d_rowsum, d_mode_w, d_c, d_err);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && max_W > 16)
      e = launch_diag_wide(d_tasks, n_tasks, n_cols, max_W, d_wire, d_phi, d_gam, gl, gr, st,
                           d_rowsum, d_mode_w, d_c, d_err, s);
    if (e != cudaSuccess) return e;
  } else {
    const size_t smem = diag_cta_bytes(max_W);
    cudaError_t e = allow_smem(diag_cta_kernel);
    if (e != cudaSuccess) return e;
    diag_cta_kernel<<<n_cols, kSweepThreads, smem, s>>>(
        d_tasks, n_tasks, n_cols, d_wire, d_phi, d_gam, reinterpret_cast<const cd*>(d_gL),
        reinterpret_cast<const cd*>(d_gR), reinterpret_cast<cd*>(d_start), d_rowsum, d_mode_w,
        d_c, d_err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const uint32_t jobs = 2 * n_cols;
  if (cols_max_W == 0) return cudaSuccess;      // every task's columns come from another kernel
  if (sizeof(C) == sizeof(cf) && cols_max_W <= 32 && d_green == nullptr)
    return launch_chain_cols(d_tasks, n_tasks, jobs, cols_max_W,
                             reinterpret_cast<const float*>(d_eta),
                             reinterpret_cast<const float*>(d_phiR), d_gam,
                             reinterpret_cast<const cf*>(d_gL), reinterpret_cast<const cf*>(d_gR),
                             reinterpret_cast<const cf*>(d_start), reinterpret_cast<float*>(d_w),
                             s);
  const size_t per = chain_warp_bytes<C>(max_W);
  int warps = warps_for(per, 8);
  if (chain_warps > 0) warps = chain_warps < chain_max<C>(max_W) ? chain_warps : chain_max<C>(max_W);
  const size_t smem = per * warps;
  if (sizeof(C) == sizeof(cd) && d_green == nullptr) {
    // two warps a CTA where the caller leaves it open, a long and a short chain, so that the
    // SMs' shares of the CTAs are the same work (eight warps a CTA 1.77 ms, two 1.67)
    if (chain_warps <= 0) warps = warps < 2 ? warps : 2;
    const size_t smem_sym = per * warps;
    const cudaError_t e = allow_smem(chain_sym_kernel);
    if (e != cudaSuccess) return e;
    chain_sym_kernel<<<(n_cols + warps - 1) / warps, 32 * warps, smem_sym, s>>>(
        d_tasks, n_tasks, n_cols, max_W, d_wire, d_phi, d_gam, reinterpret_cast<const cd*>(d_gL),
        reinterpret_cast<const cd*>(d_gR), reinterpret_cast<const cd*>(d_start),
        reinterpret_cast<double*>(d_w));
    return cudaGetLastError();
  }
  const cudaError_t e = allow_smem(chain_kernel<C>);
  if (e != cudaSuccess) return e;
  chain_kernel<C><<<(jobs + warps - 1) / warps, 32 * warps, smem, s>>>(
      d_tasks, n_tasks, jobs, max_W, d_eta, d_phiR, d_gam, d_gL, d_gR, d_start, d_w, d_green,
      d_gphi);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_lead_modes(const TaskDesc* d_tasks, int n_tasks, int max_W,
                              const double* d_wire, double* d_phi, float* d_phi32,
                              float* d_eta32, cd* d_sig, double* d_gam, int32_t* d_err,
                              cudaStream_t s) {
  if (n_tasks == 0) return cudaSuccess;
  lead_modes_kernel<<<n_tasks, 128, 0, s>>>(d_tasks, n_tasks, d_wire, d_phi, d_phi32, d_eta32,
                                            d_sig, d_gam, d_err);
  return cudaGetLastError();
}

cudaError_t launch_rgf_sweep(const TaskDesc* d_tasks, int n_tasks, int max_W, int precision,
                             const double* d_wire, const double* d_phi, const cd* d_sig,
                             void* d_gL, void* d_gR, int32_t* d_err, cudaStream_t s) {
  if (n_tasks == 0) return cudaSuccess;
  cudaError_t e;
  if (precision == NEGF_FP64) {
    e = lead_blocks(d_tasks, n_tasks, max_W, d_phi, d_sig, static_cast<cd*>(d_gL), s);
    return e != cudaSuccess ? e
                            : sweep_fp64(d_tasks, n_tasks, max_W, d_wire, static_cast<cd*>(d_gL),
                                         static_cast<cd*>(d_gR), d_err, s);
  }
  e = max_W > kOwnLeadW
          ? lead_blocks(d_tasks, n_tasks, max_W, d_phi, d_sig, static_cast<cf*>(d_gL), s)
          : cudaSuccess;
  return e != cudaSuccess ? e
                          : sweep_fp32(d_tasks, n_tasks, max_W, d_wire, d_phi, d_sig,
                                       static_cast<cf*>(d_gL), static_cast<cf*>(d_gR), d_err, s);
}

cudaError_t launch_block_columns(const TaskDesc* d_tasks, int n_tasks, uint32_t n_cols,
                                 int max_W, int precision, const double* d_wire,
                                 const float* d_eta32, const double* d_phi, const float* d_phi32,
                                 const double* d_gam, const void* d_gL,
                                 const void* d_gR, void* d_start, void* d_weights,
                                 double* d_rowsum, double* d_mode_w, double* d_c, int32_t* d_err,
                                 void* d_green, void* d_gphi, cudaStream_t s, int chain_warps,
                                 int cols_max_W) {
  if (n_tasks == 0 || n_cols == 0) return cudaSuccess;
  if (cols_max_W < 0) cols_max_W = max_W;
  if (precision == NEGF_FP64)
    return columns_impl<cd>(d_tasks, n_tasks, n_cols, max_W, d_wire, d_wire, d_phi, d_phi, d_gam,
                            static_cast<const cd*>(d_gL),
                            static_cast<const cd*>(d_gR), static_cast<cd*>(d_start),
                            static_cast<double*>(d_weights), d_rowsum, d_mode_w, d_c, d_err,
                            static_cast<cd*>(d_green), static_cast<cd*>(d_gphi), s,
                            chain_warps, cols_max_W);
  return columns_impl<cf>(d_tasks, n_tasks, n_cols, max_W, d_wire, d_eta32, d_phi, d_phi32, d_gam,
                          static_cast<const cf*>(d_gL),
                          static_cast<const cf*>(d_gR), static_cast<cf*>(d_start),
                          static_cast<float*>(d_weights), d_rowsum, d_mode_w, d_c, d_err,
                          static_cast<cf*>(d_green), static_cast<cf*>(d_gphi), s,
                          chain_warps, cols_max_W);
}

int chain_warps_max(int max_W, int precision) {
  return precision == NEGF_FP64 ? chain_max<cd>(max_W) : chain_max<cf>(max_W);
}

}  // namespace negf
