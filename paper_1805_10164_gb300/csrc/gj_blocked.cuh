// Blocked Gauss-Jordan inversion of a complex64 W x W block (16 < W <= 64) by one CTA, for the
// RGF sweeps and the diagonal blocks on slices where every site dephases (no pivot search; see
// gj_rows in k_rgf.cu for why that is safe).
//
// What bounds it: a sweep is a serial chain of inversions on a few SMs, so the time of one
// inversion is what counts.  One pivot at a time (cta_gj) needs two barriers and ~150
// instructions a warp per pivot; at W = 64 that took 67 us a slice.  Here four pivots make a
// panel, and one barrier serves a panel:
//   * the panel warps (a lane a row) bring the next panel's four columns up to date with the
//     current panel, pass its four pivot rows around, eliminate that 4 x 4 block - every lane
//     for itself, which costs no exchange within the serial chain of reciprocals - and then
//     their own rows, and publish the four pivot columns f_k (at time k) and the reciprocals;
//   * meanwhile the column warps apply the current panel to every other column: a thread owns
//     one column and up to eight rows, forms its column's four t_k = a_kj / a_kk from the four
//     pivot rows, and updates its entries four rows at a time.  The block is read from one of
//     two buffers and written to the other, so no thread waits for another within a panel.
// Each entry sees the same operations in the same order as in cta_gj
//   a_kk <- 1/a_kk;  a_kj <- t = a_kj / a_kk;  a_ik <- -a_ik / a_kk;  a_ij <- a_ij - a_ik t
// for k = 0, 1, ..., each rounding written out (bg_mul, bg_sub, bg_col), so the inverse does not
// depend on how a compiler contracts the expressions and stays what cta_gj gives.
// Measured at W = 64: 67 us a slice with one pivot at a time; 26 with one panel warp of two rows
// a lane and the pivot row broadcast by shuffles; 24 as it is.  Updates as (re, im) pairs
// (f32x2, two columns a thread, half the warps) measured 30: too few warps to hide the latencies.
#pragma once

#include <cuda_runtime.h>

#include "gj.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

constexpr int kBgPitch = 65;                  // row pitch: rows and columns free of conflicts
constexpr int kBgGroups = 8;                  // row groups of the column warps

// NH halves of 32 columns: W <= 32 -> 1, W <= 64 -> 2.  Warps 0 .. NH - 1 are the panel warps; the
// column units (half, row group) go to warps so that the schedulers (warp mod 4) with a panel
// warp, whose chain issues as much as two units, hold fewer of them.
template <int NH> constexpr int kBgThreads = NH == 2 ? 20 * 32 : 12 * 32;
template <int NH>
__device__ __forceinline__ int bg_unit(int warp) {
  if (NH == 2) {
    if (warp & 2) return (warp >> 2) * 2 + (warp & 1);            // 2, 3, 6, 7, .. 19 -> 0 .. 9
    return warp >= 4 && warp < 16 ? 8 + (warp >> 2) * 2 + (warp & 1) : -1;   // -> 10 .. 15
  }
  // 1, 2, 3, 5, 6, 7, 9, 10 -> 0 .. 7
  return (warp & 3) && warp < 11 ? (warp >> 2) * 3 + (warp & 3) - 1 : -1;
}
// the warps without columns that fetch the next slice's diagonal (its half h), -1 otherwise
template <int NH>
__device__ __forceinline__ int bg_side(int warp) {
  if (NH == 2) return warp == 16 ? 0 : warp == 17 ? 1 : -1;
  return warp == 8 ? 0 : -1;
}

// a b, a - b c, -(b c), 1 / a with every rounding explicit
__device__ __forceinline__ cf bg_mul(cf a, cf b) {
  return cf{__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x))};
}
__device__ __forceinline__ cf bg_sub(cf a, cf b, cf c) {
  const cf p = bg_mul(b, c);
  return cf{__fsub_rn(a.x, p.x), __fsub_rn(a.y, p.y)};
}
__device__ __forceinline__ cf bg_col(cf b, cf c) {
  return cf{__fmaf_rn(b.y, c.y, -__fmul_rn(b.x, c.x)),
            -__fmaf_rn(b.x, c.y, __fmul_rn(b.y, c.x))};
}
__device__ __forceinline__ cf bg_inv(cf a) {
  const float n = __fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y));
  return cf{__fdiv_rn(a.x, n), __fdiv_rn(-a.y, n)};
}

struct BgShared {
  cf B[2][64 * kBgPitch];       // the block, ping-pong
  float4 F[2][64][2];           // pivot columns f_q of a panel, a row's four together
  float4 t[2][4][2];            // per panel warp: the current panel's t_q of the next columns
  float4 blk[4][2];             // the next panel's pivot rows
  cf inv[2][4];                 // reciprocals of the panel's pivots
  cf diag[2][64];               // diagonal of E - H - Sigma_s of a slice
  int undephased[2][2];         // nonzero: the slice (half of it) has a site without dephasing
  int perm[64];                 // pivoted inversions
  int bad;                      // some inversion met a pivot without a finite reciprocal: read it
                                // after the last one only (warp 0 may set it in the next one's
                                // first panel while other warps leave this one)
};

__device__ __forceinline__ void bg_put4(float4* dst, const cf (&v)[4]) {
  dst[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  dst[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}
__device__ __forceinline__ void bg_get4(const float4* src, cf (&v)[4]) {
  const float4 a = src[0], b = src[1];
  v[0] = cf{a.x, a.y};
  v[1] = cf{a.z, a.w};
  v[2] = cf{b.x, b.y};
  v[3] = cf{b.z, b.w};
}
// The panel warps' own barrier
template <int NH>
__device__ __forceinline__ void bg_panel_sync() {
  if (NH == 1) __syncwarp();
  else asm volatile("bar.sync 1, 64;\n" ::: "memory");
}

// Panel warps: eliminate the nb pivots k1 .. k1 + nb - 1 within the panel's columns v of this
// lane's row, leaving the pivot columns in f and the reciprocals in inv; publishes them in
// buffer buf and the panel's columns, now as after these pivots, in Bout.
// kFull: nb = 4 (every panel but perhaps the last), without branches between the pivots.
template <int NH, bool kFull>
__device__ __forceinline__ void bg_factor(BgShared& S, int k1, int nb, int buf, cf* Bout,
                                          cf (&v)[4], cf (&f)[4], cf (&inv)[4]) {
  const int row = threadIdx.x;                      // panel warps are warps 0 .. NH - 1
  const int own = row - k1;                         // 0 .. 3: this lane's row is pivot row `own`
  if ((unsigned)own < 4u) bg_put4(S.blk[own], v);
  bg_panel_sync<NH>();
  // the 4 x 4 block: t_q and 1 / a_kk of each pivot, from the rows below it only
  cf D[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r) bg_get4(S.blk[r], D[r]);
  bool bad = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (kFull || q < nb) {
      const cf iv = bg_inv(D[q][q]);
      bad |= !finite_c(iv);
      inv[q] = iv;
#pragma unroll
      for (int c = 0; c < 4; ++c) D[q][c] = c == q ? iv : bg_mul(D[q][c], iv);    // t_q
#pragma unroll
      for (int r = q + 1; r < 4; ++r) {
        const cf fr = D[r][q];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          D[r][c] = c == q ? bg_col(fr, iv) : bg_sub(D[r][c], fr, D[q][c]);
      }
    }
  }
  // this lane's row
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (kFull || q < nb) {
      const cf fq = v[q];
      f[q] = fq;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const cf n = c == q ? bg_col(fq, inv[q]) : bg_sub(v[c], fq, D[q][c]);
        v[c] = own == q ? D[q][c] : n;
      }
    }
  }
  bg_put4(S.F[buf][row], f);
#pragma unroll
  for (int c = 0; c < 4; ++c) Bout[row * kBgPitch + k1 + c] = v[c];
  if (row == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) S.inv[buf][q] = inv[q];
    if (bad) S.bad = 1;
  }
}

// Invert the block.  On entry the columns >= 4 are in S.B[0], panel 0 has been eliminated by
// bg_factor (buffer 0, columns in S.B[1]; the panel warps' f and inv from it), and the CTA has
// synchronised.  On return (synchronised) the inverse is in S.B[NP & 1], NP = ceil(W / 4);
// S.bad is set (and stays so) if some pivot had no finite reciprocal; the inverse then holds no
// numbers.  side() is called by the warps without rows during panel 0.
template <int NH, typename Side>
__device__ __forceinline__ void bg_invert(BgShared& S, int W, cf (&v)[4], cf (&f)[4], cf (&inv)[4],
                                          Side side) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = bg_unit<NH>(warp);
  const int j = NH == 2 ? (unit & 1) * 32 + lane : lane;
  const int g = NH == 2 ? unit >> 1 : unit;
  const int NP = (W + 3) >> 2;
  for (int p = 0; p < NP; ++p) {
    const int k0 = 4 * p, k1 = k0 + 4, b = p & 1;
    cf* X = S.B[b];
    cf* Y = S.B[b ^ 1];
    if (warp < NH) {
      if (p + 1 < NP) {
        // panel p (four pivots, since another follows) applied to the columns of panel p + 1:
        // t_q of column lane & 3, exchanged through shared memory, then this lane's row
        const int row = threadIdx.x;
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = X[row * kBgPitch + k1 + c];
        const int c0 = lane & 3;
        cf R[4], t[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) R[r] = X[(k0 + r) * kBgPitch + k1 + c0];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          t[q] = bg_mul(R[q], inv[q]);
#pragma unroll
          for (int r = q + 1; r < 4; ++r) {
            const float4 ff = S.F[b][k0 + r][q >> 1];
            R[r] = bg_sub(R[r], q & 1 ? cf{ff.z, ff.w} : cf{ff.x, ff.y}, t[q]);
          }
        }
        cf* ts = reinterpret_cast<cf*>(S.t[warp]);
        if (lane < 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) ts[4 * q + lane] = t[q];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          cf tq[4];
          bg_get4(S.t[warp][q], tq);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const cf n = bg_sub(v[c], f[q], tq[c]);
            v[c] = row == k0 + q ? tq[c] : n;
          }
        }
        if (W - k1 >= 4) bg_factor<NH, true>(S, k1, 4, b ^ 1, X, v, f, inv);
        else bg_factor<NH, false>(S, k1, W - k1, b ^ 1, X, v, f, inv);
      }
    } else if (unit >= 0) {
      const int nb = min(4, W - k0);
      const bool act = j < W && (j >> 2) != p && (j >> 2) != p + 1;
      // the t_q of this column; with fewer than four pivots left the rest come from rows >= W
      // and are not used
      cf R[4], t[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) R[r] = X[(k0 + r) * kBgPitch + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        t[q] = bg_mul(R[q], S.inv[b][q]);
#pragma unroll
        for (int r = q + 1; r < 4; ++r) {
          const float4 ff = S.F[b][k0 + r][q >> 1];
          R[r] = bg_sub(R[r], q & 1 ? cf{ff.z, ff.w} : cf{ff.x, ff.y}, t[q]);
        }
      }
      if (nb == 4) {
        // the rows that hold no pivot of this panel, four at a time (rows >= W are computed
        // from whatever the buffer holds and not stored)
#pragma unroll
        for (int rc = 0; rc < 8; rc += 4) {
          if (g + kBgGroups * rc < W) {
            cf a[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int i = g + kBgGroups * (rc + r);
              a[r] = X[i * kBgPitch + j];
              cf fi[4];
              bg_get4(S.F[b][i], fi);
#pragma unroll
              for (int q = 0; q < 4; ++q) a[r] = bg_sub(a[r], fi[q], t[q]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int i = g + kBgGroups * (rc + r);
              if (act && i < W && (unsigned)(i - k0) >= 4u) Y[i * kBgPitch + j] = a[r];
            }
          }
        }
      } else {
        for (int i = g; i < k0; i += kBgGroups) {
          cf a = X[i * kBgPitch + j];
          cf fi[4];
          bg_get4(S.F[b][i], fi);
#pragma unroll
          for (int q = 0; q < 3; ++q)
            if (q < nb) a = bg_sub(a, fi[q], t[q]);
          if (act) Y[i * kBgPitch + j] = a;
        }
      }
      // the pivot row of this group, if it has one: t at its own pivot, updated by the others
      const int own = (g - k0) & (kBgGroups - 1);
      if (own < nb) {
        const int i = k0 + own;
        cf a = X[i * kBgPitch + j];
        cf fi[4];
        bg_get4(S.F[b][i], fi);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < nb) a = q == own ? t[q] : bg_sub(a, fi[q], t[q]);
        if (act) Y[i * kBgPitch + j] = a;
      }
    } else if (p == 0) {
      side();
    }
    __syncthreads();
  }
}

// The buffer of S.B in which bg_pivoted takes its block (one exchange of buffers per pivot, and
// one as the result is put in order)
__device__ __forceinline__ cf* bg_pivoted_in(BgShared& S, int W) {
  return S.B[((((W + 3) >> 2) & 1) ^ 1) ^ (W & 1)];
}

// Invert the W x W block in bg_pivoted_in (pitch kBgPitch) with partial pivoting into S.B[NP & 1]:
// what cta_gj does, in the same order and rounding, so the same inverse.  Slices with a site
// without dephasing take it.  A pivot's latency bounds it, so every warp finds the pivot for
// itself, every thread forms the reciprocal and the exchanged rows as it reads them, and the
// block is read from one buffer and written to the other: one barrier a pivot, where cta_gj has
// five.  The columns are put in order on the way out.  Synchronised before and after; false
// (uniformly) on a zero or non-finite pivot.  GB300, every third site undephased, sweeps: W=64 x
// L=100, 8 energies 12.7 -> 7.4 ms, W=40 x L=50, 16 energies 2.67 -> 1.46, W=32 x L=100, 32 energies
// 3.99 -> 1.94 (cta_gj by the panels' 640 or 384 threads was slower than by the 1024 threads that
// sweeps had before the panels: W=64 x L=60 6.1 ms against 7.5).
__device__ __forceinline__ bool bg_pivoted(BgShared& S, int W) {
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31;
  const int j = tid % W, g = tid / W, G = blockDim.x / W;   // this thread's column and row group
  cf* X = bg_pivoted_in(S, W);
  cf* Y = X == S.B[0] ? S.B[1] : S.B[0];
  for (int k = 0; k < W; ++k) {
    // the row p >= k with the largest |a_pk|, the first of equals; non-negative floats order like
    // their bits, and a NaN is never the largest
    const int i0 = k + lane, i1 = i0 + 32;
    const float v0 = i0 < W ? norm2(X[i0 * kBgPitch + k]) : 0.f;
    const float v1 = i1 < W ? norm2(X[i1 * kBgPitch + k]) : 0.f;
    const unsigned b0 = v0 > 0.f ? __float_as_uint(v0) : 0u, b1 = v1 > 0.f ? __float_as_uint(v1) : 0u;
    const unsigned best = __reduce_max_sync(FULL, b0 > b1 ? b0 : b1);
    const unsigned at0 = __ballot_sync(FULL, b0 == best), at1 = __ballot_sync(FULL, b1 == best);
    if (best == 0u || best >= 0x7f800000u) return false;    // zero, infinite or no number at all
    const int p = at0 ? k + __ffs(at0) - 1 : k + 32 + __ffs(at1) - 1;
    if (tid == 0) S.perm[k] = p;
    const cf inv = cdiv(cf{1.f, 0.f}, X[p * kBgPitch + k]);
    if (!finite_c(inv)) return false;
    if (g < G) {
      const cf t = j == k ? inv : bg_mul(X[p * kBgPitch + j], inv);        // a_kj / a_kk
      for (int i = g; i < W; i += G) {
        const int from = i == p ? k : i;                    // rows k and p exchanged
        const cf f = X[from * kBgPitch + k];
        cf v;
        if (i == k) v = t;
        else if (j == k) v = bg_col(f, inv);
        else v = bg_sub(X[from * kBgPitch + j], f, t);
        Y[i * kBgPitch + j] = v;
      }
    }
    __syncthreads();
    cf* const Z = X;
    X = Y;
    Y = Z;
  }
  // the exchanges of rows undone as exchanges of columns, in reverse order: column j goes to `at`
  if (g < G) {
    int at = j;
    for (int k = W - 1; k >= 0; --k) {
      const int p = S.perm[k];
      at = at == k ? p : at == p ? k : at;
    }
    for (int i = g; i < W; i += G) Y[i * kBgPitch + at] = X[i * kBgPitch + j];
  }
  __syncthreads();
  return true;
}

// Form a slice's block, entry (i, c) = form(i, c), and invert it; the inverse is in S.B[NP & 1] on
// return (synchronised).  form may read entry (i, c) of the block before, which is in S.B[NP & 1].
// pivot: partial pivoting (the slice has a site without dephasing); false (uniformly) if a pivot
// then has no finite reciprocal, without pivoting see S.bad.  side() is called by the warps without
// columns.
template <int NH, typename Form, typename Side>
__device__ __forceinline__ bool bg_slice(BgShared& S, int W, bool pivot, Form form, Side side) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NP = (W + 3) >> 2;
  if (__builtin_expect(!pivot, 1)) {
    const int unit = bg_unit<NH>(warp);
    const int j = NH == 2 ? (unit & 1) * 32 + lane : lane;
    const int g = NH == 2 ? unit >> 1 : unit;
    cf v[4], f[4], inv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[c] = inv[c] = cf{0.f, 0.f};
    if (warp < NH) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (tid < W && c < W) v[c] = form(tid, c);
      if (W >= 4) bg_factor<NH, true>(S, 0, 4, 0, S.B[1], v, f, inv);
      else bg_factor<NH, false>(S, 0, W, 0, S.B[1], v, f, inv);
    } else if (unit >= 0 && j >= 4 && j < W) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int i = g + kBgGroups * r;
        if (i < W) S.B[0][i * kBgPitch + j] = form(i, j);
      }
    }
    __syncthreads();
    bg_invert<NH>(S, W, v, f, inv, side);
    return true;
  }
  cf* A = bg_pivoted_in(S, W);
  for (int idx = tid; idx < W * W; idx += blockDim.x)
    A[idx / W * kBgPitch + idx % W] = form(idx / W, idx % W);
  side();
  __syncthreads();
  return bg_pivoted(S, W);
}

}  // namespace
}  // namespace negf
