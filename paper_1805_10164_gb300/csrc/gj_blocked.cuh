// Blocked Gauss-Jordan inversion of a complex64 W x W block (16 < W <= 64) by one CTA, for the
// RGF sweeps and the diagonal blocks on slices where every site dephases (no pivot search; see
// gj_rows in k_rgf.cu for why that is safe).
//
// What bounds it: a sweep is a serial chain of inversions on a few SMs, so the time of one
// inversion is what counts.  One pivot at a time (cta_gj) needs two barriers and ~150
// instructions a warp per pivot; at W = 64 that took 67 us a slice.  Here four pivots make a
// panel, and one barrier serves a panel:
//   * warp 0 (the panel warp) holds the next panel's columns in registers, a lane two rows: it
//     applies the current panel's four pivots to them, then eliminates within the panel, the
//     pivot row broadcast by shuffles.  It publishes the four pivot columns f_k (at time k) and
//     the reciprocals;
//   * meanwhile the other warps apply the current panel to every other column: a thread owns
//     one column and up to eight rows, forms its column's four t_k = a_kj / a_kk from the four
//     pivot rows, and updates its entries from registers.  The block is read from one of two
//     buffers and written to the other, so no thread waits for another within a panel.
// Each entry sees the same operations in the same order as in cta_gj
//   a_kk <- 1/a_kk;  a_kj <- t = a_kj / a_kk;  a_ik <- -a_ik / a_kk;  a_ij <- a_ij - a_ik t
// for k = 0, 1, ..., each rounding written out (bg_mul, bg_sub, bg_col), so the inverse does not
// depend on how a compiler contracts the expressions and stays what cta_gj gives.
//
// The panel warp shares its scheduler (warps 0, 4, 8, ...) with fewer column warps than the
// other three schedulers hold: its serial chain is as long as the other warps' work.
#pragma once

#include <cuda_runtime.h>

#include "gj.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

constexpr int kBgPitch = 65;                  // row pitch: rows and columns free of conflicts
constexpr int kBgGroups = 8;                  // row groups of the column warps

// NH halves of 32 columns: W <= 32 -> 1, W <= 64 -> 2.
template <int NH> constexpr int kBgThreads = NH == 2 ? 19 * 32 : 11 * 32;
// column unit (half, row group) of a warp, -1 for the panel warp and the warps that only keep
// the schedulers balanced
template <int NH>
__device__ __forceinline__ int bg_unit(int warp) {
  if (NH == 1) return (warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 : -1;   // 1,2,3,5,6,7,9,10
  if (warp >= 17) return warp - 3;                                        // 17, 18 -> 14, 15
  if (warp & 3) return (warp >> 2) * 3 + (warp & 3) - 1;                  // 0 .. 11
  return warp == 4 ? 12 : warp == 8 ? 13 : -1;
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
  cf inv[2][4];                 // reciprocals of the panel's pivots
  cf t[4][4];                   // the current panel's t_q of the next panel's columns
  cf diag[2][64];               // diagonal of E - H - Sigma_s of a slice
  int undephased[2][2];         // nonzero: the slice (half of it) has a site without dephasing
  int perm[64];                 // pivoted fallback
  int flag[2];
  int bad;                      // a pivot without a finite reciprocal
};

// Eliminate the nb pivots k1 .. k1 + nb - 1 within the panel's columns v (lane's rows lane and
// lane + 32), leaving the pivot columns in f and the reciprocals in inv; publishes them in
// buffer buf and the panel's columns, now as after these pivots, in Bout.
template <int NH>
__device__ __forceinline__ void bg_factor(BgShared& S, int k1, int nb, int buf, cf* Bout,
                                          cf (&v)[NH][4], cf (&f)[NH][4], cf (&inv)[4]) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  bool bad = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q < nb) {
      const int k = k1 + q, src = k & 31;
      cf r[4];
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const int c = (q + cc) & 3;                        // the pivot first
        const cf own = NH == 2 && k >= 32 ? v[NH - 1][c] : v[0][c];
        r[c].x = __shfl_sync(FULL, own.x, src);
        r[c].y = __shfl_sync(FULL, own.y, src);
      }
      const cf iv = bg_inv(r[q]);
      bad |= !finite_c(iv);
      cf t[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) t[c] = c == q ? iv : bg_mul(r[c], iv);
#pragma unroll
      for (int m = 0; m < NH; ++m) {
        const bool me = lane + 32 * m == k;
        const cf fm = v[m][q];
        f[m][q] = fm;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const cf n = c == q ? bg_col(fm, iv) : bg_sub(v[m][c], fm, t[c]);
          v[m][c] = me ? t[c] : n;
        }
      }
      inv[q] = iv;
    }
  }
#pragma unroll
  for (int m = 0; m < NH; ++m) {
    const int row = lane + 32 * m;
    S.F[buf][row][0] = make_float4(f[m][0].x, f[m][0].y, f[m][1].x, f[m][1].y);
    S.F[buf][row][1] = make_float4(f[m][2].x, f[m][2].y, f[m][3].x, f[m][3].y);
#pragma unroll
    for (int c = 0; c < 4; ++c) Bout[row * kBgPitch + k1 + c] = v[m][c];
  }
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) S.inv[buf][q] = inv[q];
    if (bad) S.bad = 1;
  }
}

// Invert the block.  On entry the columns >= 4 are in S.B[0], panel 0 has been eliminated by
// bg_factor (buffer 0, columns in S.B[1]; the panel warp's f and inv from it), and the CTA has
// synchronised.  On return (synchronised) the inverse is in S.B[NP & 1], NP = ceil(W / 4);
// S.bad is set if some pivot had no finite reciprocal.  side(p) is called by the warps without
// columns during panel 0.
template <int NH, typename Side>
__device__ __forceinline__ void bg_invert(BgShared& S, int W, cf (&v)[NH][4], cf (&f)[NH][4],
                                          cf (&inv)[4], Side side) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = bg_unit<NH>(warp);
  const int NP = (W + 3) >> 2;
  const int j = NH == 2 ? (unit & 1) * 32 + lane : lane;
  const int g = NH == 2 ? unit >> 1 : unit;
  for (int p = 0; p < NP; ++p) {
    const int k0 = 4 * p, k1 = k0 + 4, b = p & 1;
    cf* X = S.B[b];
    cf* Y = S.B[b ^ 1];
    if (warp == 0) {
      if (p + 1 < NP) {
        // panel p (four pivots, since another follows) applied to the columns of panel p + 1
#pragma unroll
        for (int m = 0; m < NH; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[m][c] = X[(lane + 32 * m) * kBgPitch + k1 + c];
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
        if (lane < 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) S.t[q][lane] = t[q];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const cf tq = S.t[q][c];
#pragma unroll
            for (int m = 0; m < NH; ++m) {
              const cf n = bg_sub(v[m][c], f[m][q], tq);
              v[m][c] = lane + 32 * m == k0 + q ? tq : n;
            }
          }
        }
        bg_factor<NH>(S, k1, min(4, W - k1), b ^ 1, X, v, f, inv);
      }
    } else if (unit >= 0) {
      const int pj = j >> 2;
      if (j < W && pj != p && pj != p + 1) {
        const int nb = min(4, W - k0);
        cf R[4], t[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) R[r] = X[(k0 + r) * kBgPitch + j];   // rows >= W: unused
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          t[q] = cf{0.f, 0.f};
          if (q < nb) {
            t[q] = bg_mul(R[q], S.inv[b][q]);
#pragma unroll
            for (int r = q + 1; r < 4; ++r) {
              const float4 ff = S.F[b][k0 + r][q >> 1];
              R[r] = bg_sub(R[r], q & 1 ? cf{ff.z, ff.w} : cf{ff.x, ff.y}, t[q]);
            }
          }
        }
        if (nb == 4) {
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int i = g + kBgGroups * r;
            if (i < W) {
              cf a = X[i * kBgPitch + j];
              const float4 f01 = S.F[b][i][0], f23 = S.F[b][i][1];
              a = bg_sub(a, cf{f01.x, f01.y}, t[0]);
              a = bg_sub(a, cf{f01.z, f01.w}, t[1]);
              a = bg_sub(a, cf{f23.x, f23.y}, t[2]);
              a = bg_sub(a, cf{f23.z, f23.w}, t[3]);
              if ((unsigned)(i - k0) >= 4u) Y[i * kBgPitch + j] = a;
            }
          }
        } else {
          for (int i = g; i < k0; i += kBgGroups) {        // the last, narrower panel
            cf a = X[i * kBgPitch + j];
            const float4 f01 = S.F[b][i][0], f23 = S.F[b][i][1];
            a = bg_sub(a, cf{f01.x, f01.y}, t[0]);
            if (nb > 1) a = bg_sub(a, cf{f01.z, f01.w}, t[1]);
            if (nb > 2) a = bg_sub(a, cf{f23.x, f23.y}, t[2]);
            Y[i * kBgPitch + j] = a;
          }
        }
        // the pivot row of this group, if it has one: t at its own pivot, updated by the others
        const int own = (g - k0) & (kBgGroups - 1);
        if (own < nb) {
          const int i = k0 + own;
          cf a = X[i * kBgPitch + j];
          const float4 f01 = S.F[b][i][0], f23 = S.F[b][i][1];
          const cf fi[4] = {cf{f01.x, f01.y}, cf{f01.z, f01.w}, cf{f23.x, f23.y},
                            cf{f23.z, f23.w}};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < nb) a = q == own ? t[q] : bg_sub(a, fi[q], t[q]);
          Y[i * kBgPitch + j] = a;
        }
      }
    } else if (p == 0) {
      side();
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace negf
