// Block-column propagation of the RGF for W = 64 slices in FP32 on the CUDA cores, one CTA per
// pair of block columns (Sec. III.B): G_{k,m} = -t g^L_k G_{k+1,m} towards slice 0 and
// G_{k,m} = -t g^R_k G_{k-1,m} towards slice L - 1, each block emitted as the Step 6' weights
// w_{(m,b),(k,a)} = eta_{k,a} |G_{k,m}[a][b]|^2 of the column's W rows (Eq. draw_i_simult) and,
// at the boundary slices, the lead weights <psi_b|Gamma|psi_b> = sum_nu Gamma_nu
// |(Phi^T G_{k,m})_{nu b}|^2.  Same weights as chain_kernel (one warp per column), the two
// columns side by side: X_k [64][128] = (-t g_k) [64][64] X_{k+1} in shared memory.
//
// What bounds it: the FP32 multiply-add pipe (64 x 64 x 128 complex products a step, 16,384
// cycles of an SM's 128 lanes).  One set of warps that first multiplies and then emits left that
// pipe idle for half of a step, so the CTA's 16 warps have two roles:
//   * warps 0..7 multiply.  A lane holds 8 x 4 outputs as (re, im) pairs and uses the paired
//     multiply-add (fma.rn.f32x2), which does not raise the pipe's rate but takes half the
//     issue slots, so that the other warps' instructions fit between.  (-t g) lies in shared
//     memory with every value twice, (x, x, y, y), so that a pair operand is one half of a
//     16-byte load; X's swapped pair (-im, re) is made in registers, twice per eight uses;
//   * warps 8..15 emit the block of the step before meanwhile, and bring in the next g.
// X is overwritten in place between two barriers at the end of a step, together with |X|^2
// (FP32, N below), from which the emitting warps form every weight.
// W = 64 uses the symmetry G = G^T (H real symmetric, every self-energy a complex symmetric
// matrix), which halves the products: only the chains towards slice 0 run (and the one of the
// lead-L injection column towards slice L - 1).  A block G_{k,m} (k < m) of site column m gives
// besides the rows (m, b) the rows (k, a) of slice k towards slice m:
// w_{(k,a),(m,b)} = eta_{m,b} |G_{(m,b),(k,a)}|^2 = eta_{m,b} |G_{k,m}[a][b]|^2, and the block
// (G Phi_R)_k of the lead-R injection column gives the lead-R weights of the rows of slice k:
// <psi|Gamma_R|psi> = sum_nu Gamma_nu |(Phi_R^T G_{L-1,k})_{nu a}|^2 = sum_nu Gamma_nu
// |(G Phi_R)_k[a][nu]|^2.  Every weight is written by exactly one job.
//
// Two-level tables of W = 64 (l2_fused): each step's blocks are the 64 weights of a (row,
// slice) pair, exactly what a level-2 block of a two-level table draws from, so the kernel
// writes the block (level2.cuh: the inverse-CDF thresholds of the slice, the same arithmetic
// as the level-2 pass) and the slice's level-1 weight instead of the weights: the rows x K
// weights are never stored or read back.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "level2.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

constexpr int kW = 64;
constexpr int kN = 2 * kW;                    // two columns side by side
constexpr int kThreads = 512;
constexpr int kMul = 256;                     // threads of the multiplying warps
constexpr int kNPitch = kN + 1;               // row pitch of N
constexpr int kB2 = 8 + kW;                   // level-2 block of a 64-site slice: guide + octets
constexpr int kSP = kB2 + 4;                  // its pitch in the staging: 16-byte aligned, and
                                              // eight blocks start on different banks
// X, two g blocks (doubled values), N
constexpr size_t kSmem = sizeof(cf) * kW * kN + 2 * sizeof(float4) * kW * kW +
                         sizeof(float) * kW * kNPitch;

// eta |G|^2 with every rounding explicit, so that the weight of a (row, site) pair has the same
// bits wherever it is formed (stored weights, or a level-2 block built in the kernel)
__device__ __forceinline__ float nsq(cf v) {
  return __fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y));
}

typedef unsigned long long f2;                // two floats: a register pair
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ ulonglong2 lds2(const void* p) {
  return *reinterpret_cast<const ulonglong2*>(p);
}

// Element (a, b') of N.  The column is permuted within groups of 32 so that the emitting
// lanes, eight rows (or columns) by four chunks of 16, read 32 different banks either way.
__device__ __forceinline__ int n_at(int a, int bp) {
  return a * kNPitch + (bp ^ (((bp >> 5) & 1) << 3) ^ (((a >> 4) & 3) << 3));
}
// Element (a, c) of the doubled -t g: the lanes that write a row and those that read a column
// take different banks.
__device__ __forceinline__ int g_at(int a, int c) { return c * kW + (a ^ (c & 7)); }

// shared -> global copy of `bytes` (a multiple of 16, both ends 16-byte aligned) by the TMA
// engine, in the calling thread's bulk group
__device__ __forceinline__ void bulk_store(void* gmem, const void* smem, unsigned bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(gmem), "r"(sa),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(kPending) : "memory");
}
__device__ __forceinline__ void fence_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// the emitting warps' own barrier
__device__ __forceinline__ void emit_sync() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(kThreads - kMul) : "memory");
}

// the whole CTA, the two roles from their own code
__device__ __forceinline__ void step_sync() {
  asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1) chain_cta_kernel(
    const TaskDesc* __restrict__ tasks, const TcJob* __restrict__ jobs,
    const float* __restrict__ eta32, const float* __restrict__ phi32,
    const double* __restrict__ gam, const cf* __restrict__ gL, const cf* __restrict__ gR,
    const cf* __restrict__ start, float* __restrict__ weights, uint64_t* __restrict__ tab,
    int32_t* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem[];
  cf* X = reinterpret_cast<cf*>(smem);                     // [c][b']
  float4* G0 = reinterpret_cast<float4*>(X + kW * kN);     // two (-t g) blocks, g_at
  float* N = reinterpret_cast<float*>(G0 + 2 * kW * kW);   // |X|^2, n_at

  const int tid = threadIdx.x, lane = tid & 31;
  const bool mul = tid < kMul;
  const int ew = (tid - kMul) >> 5;                        // emitting warp 0..7
  const TcJob job = jobs[blockIdx.x];
  const TaskDesc d = tasks[job.task];
  const int L = d.L, n = d.n, K = d.K;
  const int dir = job.dir;
  auto m0_of = [&](int yy) { return yy < L ? yy : (yy == L ? 0 : L - 1); };
  const int ys[2] = {job.y0, job.y1};
  const float mt = (float)(-d.t);
  const float* eta = eta32 + d.onsite_off / 2;
  const cf* gsrc = (dir == 0 ? gL : gR) + d.g_off;
  float* wt = weights + d.wt_off;
  const bool fused = d.l2_fused != 0;
  float* l1 = weights + d.l1w_off;                         // fused: level-1 weights [rows][L+2]
  uint32_t* l2 = reinterpret_cast<uint32_t*>(tab + d.tab_off);   // fused: [rows][L][kB2]
  bool bad = false;
  auto row_of = [&](int y, int b) -> uint64_t {
    return y < L ? (uint64_t)y * kW + b : (uint64_t)n + (uint64_t)(y - L) * kW + b;
  };
  // Fused: the level-2 blocks of 64 rows (row0 + r) towards `slice` from 64 weights each,
  // e(i) N(r, i); emitting warp ew builds rows 8 ew .. 8 ew + 7, lane (q, r) chunk q of row
  // 8 ew + r, stages the blocks in stg (this warp's) and sends each off as one bulk copy.
  auto put_blocks = [&](uint32_t* stg, const float* e, uint64_t row0, int slice, auto norm) {
    const int q = lane >> 3, r = lane & 7;
    float w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i)
      w[i] = __fmul_rn(__ldg(e + 16 * q + i), norm(8 * ew + r, 16 * q + i));
    uint32_t c[16];
    float tot = 0.f;
    bad |= !level2_fp32_quad(w, q, c, &tot);
    const uint64_t row = row0 + 8 * ew + r;
    if (q == 3) c[15] = kCdfOne;                           // the slice's last threshold
    uint32_t* dst = stg + r * kSP;
    *reinterpret_cast<uint2*>(dst + 2 * q) = make_uint2(c[7], c[15]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<uint4*>(dst + 8 + 16 * q + 4 * i) =
          make_uint4(c[4 * i], c[4 * i + 1], c[4 * i + 2], c[4 * i + 3]);
    fence_async_shared();
    __syncwarp();
    if (q == 0) {
      l1[row * (L + 2) + slice] = tot;
      bulk_store(l2 + (row * L + slice) * kB2, dst, kB2 * 4);
      bulk_commit();
    }
  };
  // Emit slice k from N (and X), by the emitting warps: the weights of the columns in `mask`,
  // and of the rows (k, a) towards the site columns in `tmask` (their slice ys[col], weights
  // eta_{y,b} |G_{k,y}[a][b]|^2).  stage: shared memory free during the call (39 KB).
  auto emit = [&](int k, unsigned mask, unsigned tmask, uint32_t* stage) {
    uint32_t* stg = stage + ew * 2 * 8 * kSP;
    int pass = 0;
    auto turn = [&]() {
      // two staging areas in turn: the copies of the one before last have been read
      uint32_t* s = stg + (pass & 1) * 8 * kSP;
      if (pass >= 2) {
        if (lane < 8) bulk_wait_read<1>();
        __syncwarp();
      }
      ++pass;
      return s;
    };
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      if (!(mask & (1u << col))) continue;
      if (fused) {
        put_blocks(turn(), eta + k * kW, row_of(ys[col], 0), k,
                   [&](int r, int a) { return N[n_at(a, col * kW + r)]; });
      } else {
        for (int r = ew; r < kW; r += 8) {
          float* dst = wt + row_of(ys[col], r) * K + (uint64_t)k * kW;
#pragma unroll
          for (int a = lane; a < kW; a += 32)
            dst[a] = __fmul_rn(__ldg(eta + k * kW + a), N[n_at(a, col * kW + r)]);
        }
      }
    }
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      if (!(tmask & (1u << col))) continue;
      const float* em = eta + ys[col] * kW;
      if (fused) {
        put_blocks(turn(), em, (uint64_t)k * kW, ys[col],
                   [&](int a, int b) { return N[n_at(a, col * kW + b)]; });
      } else {
        for (int a = ew; a < kW; a += 8) {
          float* dst = wt + (uint64_t)(k * kW + a) * K + (uint64_t)ys[col] * kW;
#pragma unroll
          for (int b = lane; b < kW; b += 32)
            dst[b] = __fmul_rn(__ldg(em + b), N[n_at(a, col * kW + b)]);
        }
      }
    }
    if (dir == 0) {
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        // lead-R weights of the rows of slice k from (G Phi_R)_k: eight threads per row
        if (!(mask & (1u << col)) || ys[col] != L + 1 || k == L - 1) continue;
        const int te = tid - kMul, q = te & 7;
        for (int a = te >> 3; a < kW; a += (kThreads - kMul) / 8) {
          float part = 0.f;
#pragma unroll
          for (int nu = q * 8; nu < q * 8 + 8; ++nu) {
            const cf v = X[a * kN + col * kW + nu];
            part = __fmaf_rn((float)gam[d.lead_off + nu],
                             __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)), part);
          }
          part += __shfl_xor_sync(0xffffffffu, part, 1);
          part += __shfl_xor_sync(0xffffffffu, part, 2);
          part += __shfl_xor_sync(0xffffffffu, part, 4);
          if (q == 0) {
            if (fused) l1[(uint64_t)(k * kW + a) * (L + 2) + L + 1] = part;
            else wt[(uint64_t)(k * kW + a) * K + n + 1] = part;
          }
        }
      }
    }
    if (lane < 8) bulk_wait_read<0>();
    __syncwarp();
  };
  // Lead weights of the columns in `mask` from X at a boundary slice k, by the whole CTA; Phi
  // (FP32) and the partial sums take the first g block, which no product needs any more (or
  // yet).  Synchronised before and after.
  auto lead_weights = [&](int k, unsigned mask) {
    float* phis = reinterpret_cast<float*>(G0);
    float* gams = phis + kW * kW;
    float* parts = gams + kW;
    for (int i = tid; i < kW * kW; i += kThreads) phis[i] = phi32[d.phi_off + i];
    for (int i = tid; i < kW; i += kThreads) gams[i] = (float)gam[d.lead_off + i];
    __syncthreads();
    const int r = tid % kN, h = tid / kN;                  // four quarters of the modes
    float part = 0.f;
    for (int nu = h * 16; nu < h * 16 + 16; ++nu) {
      float zr = 0.f, zi = 0.f;
      for (int a = 0; a < kW; ++a) {
        const float p = phis[a * kW + nu];
        const cf v = X[a * kN + r];
        zr = __fmaf_rn(p, v.x, zr);
        zi = __fmaf_rn(p, v.y, zi);
      }
      part = __fmaf_rn(gams[nu], __fmaf_rn(zr, zr, __fmul_rn(zi, zi)), part);
    }
    parts[h * kN + r] = part;
    __syncthreads();
    if (h == 0) {
      const int col = r / kW;
      if (mask & (1u << col)) {
        const float lw = (parts[r] + parts[kN + r]) + (parts[2 * kN + r] + parts[3 * kN + r]);
        const uint64_t row = row_of(ys[col], r % kW);
        if (fused) {
          if (k == 0) l1[row * (L + 2) + L] = lw;
          if (k == L - 1) l1[row * (L + 2) + L + 1] = lw;
        } else {
          if (k == 0) wt[row * K + n] = lw;
          if (k == L - 1) wt[row * K + n + 1] = lw;
        }
      }
    }
    __syncthreads();
  };
  // start block of column slot col into X[:, col*64 .. col*64+63]
  auto load_start = [&](int col) {
    const cf* st = start + d.start_off + (uint64_t)ys[col] * kW * kW;
    for (int i = tid; i < kW * kW; i += kThreads)
      X[(i / kW) * kN + col * kW + i % kW] = st[i];
  };

  unsigned have = 0;
  for (int col = 0; col < 2; ++col)
    if (ys[col] >= 0) have |= 1u << col;
  // direction 0 emits every column's start slice
  if (dir == 0) {
    for (int col = 0; col < 2; ++col) {
      if (!(have & (1u << col))) continue;
      const int m0 = m0_of(ys[col]);
      load_start(col);
      __syncthreads();
      for (int i = tid; i < kW * kW; i += kThreads) {
        const int a = i / kW, b = col * kW + i % kW;
        N[n_at(a, b)] = nsq(X[a * kN + b]);
      }
      __syncthreads();
      if (m0 == 0 || m0 == L - 1) lead_weights(m0, 1u << col);
      if (!mul) emit(m0, 1u << col, 0u, reinterpret_cast<uint32_t*>(G0));
      __syncthreads();
    }
  }
  const int m0a = m0_of(job.y0), m0b = job.y1 >= 0 ? m0_of(job.y1) : m0a;
  const int k_first = dir == 0 ? max(m0a, m0b) - 1 : min(m0a, m0b) + 1;
  const int k_end = dir == 0 ? -1 : L;
  const int kstep = dir == 0 ? -1 : 1;
  // -t g_k, doubled, into G (threads t0, t0 + nt, ...)
  auto put_g = [&](int k, float4* G, int t0, auto nt) {
    constexpr int kPer = kW * kW / decltype(nt)::value;
    const cf* gk = gsrc + (uint64_t)k * kW * kW;
    cf v[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) v[q] = gk[t0 + q * decltype(nt)::value];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = t0 + q * decltype(nt)::value;
      const float gx = mt * v[q].x, gy = mt * v[q].y;
      G[g_at(i / kW, i % kW)] = make_float4(gx, gx, gy, gy);
    }
  };
  if (k_first != k_end) put_g(k_first, G0, tid, std::integral_constant<int, kThreads>());
  // multiplying lane: rows a = 32 wa + ty + 4 i, columns b' = 32 wb + 2 tx + 16 h (+ 1)
  const int ty = lane >> 3, tx = lane & 7, mw = tid >> 5;
  const int wa = mw & 1, wb = (mw >> 1) & 3;
  int k_prev = -1, buf = 0;
  unsigned act_prev = 0, t_prev = 0;
  for (int k = k_first; k != k_end; k += kstep) {
    unsigned active = 0;
    for (int col = 0; col < 2; ++col) {
      if (!(have & (1u << col))) continue;
      const int m0 = m0_of(ys[col]);
      if (dir == 0 ? k < m0 : k > m0) active |= 1u << col;
      if (dir == 0 ? k == m0 - 1 : k == m0 + 1) load_start(col);
    }
    if (active != act_prev) __syncthreads();               // a column has joined
    if (mul) {
      const float4* G = G0 + buf * kW * kW + 32 * wa;
      const cf* Xl = X + 32 * wb + 2 * tx;
      f2 acc[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 1
      for (int c0 = 0; c0 < kW; c0 += 8) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int c = c0 + s;
          const ulonglong2 xa = lds2(Xl + c * kN), xb = lds2(Xl + c * kN + 16);
          const f2 x[4] = {xa.x, xa.y, xb.x, xb.y};
          f2 xs[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 v = unpack2(x[j]);
            xs[j] = pack2(-v.y, v.x);
          }
          const float4* Gc = G + c * kW + (ty ^ (s & 3));
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const ulonglong2 g = lds2(Gc + ((4 * i) ^ (s & 4)));
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fma2(g.x, x[j], acc[i][j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fma2(g.y, xs[j], acc[i][j]);
          }
        }
      }
      step_sync();                                         // X and N have been read
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int a = 32 * wa + ty + 4 * i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int b = 32 * wb + 2 * tx + 16 * h;
          *reinterpret_cast<ulonglong2*>(X + a * kN + b) =
              make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
          const float2 u = unpack2(acc[i][2 * h]), v = unpack2(acc[i][2 * h + 1]);
          N[n_at(a, b)] = nsq(cf{u.x, u.y});
          N[n_at(a, b + 1)] = nsq(cf{v.x, v.y});
        }
      }
    } else {
      float4* Gn = G0 + (buf ^ 1) * kW * kW;
      if (k_prev >= 0) {
        emit(k_prev, act_prev, t_prev, reinterpret_cast<uint32_t*>(Gn));
        emit_sync();                                       // the staging has been read
      }
      if (k + kstep != k_end)
        put_g(k + kstep, Gn, tid - kMul, std::integral_constant<int, kThreads - kMul>());
      step_sync();
    }
    __syncthreads();
    if (k == 0 || k == L - 1) lead_weights(k, active);     // the last step of its direction
    k_prev = k;
    act_prev = active;
    t_prev = 0;
    if (dir == 0)
      for (int col = 0; col < 2; ++col)
        if ((active & (1u << col)) && ys[col] < L) t_prev |= 1u << col;
    buf ^= 1;
  }
  if (!mul && k_prev >= 0) emit(k_prev, act_prev, t_prev, reinterpret_cast<uint32_t*>(G0));
  if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERR_NONFINITE);
}

// ---- 16 < W <= 32: the same recursion with the pair's 2W columns side by side --------------
// One CTA of 128 threads per job (four CTAs fit an SM): X_k [W][2W] = (-t g_k) [W][W] X_{k+1}
// in shared memory, thread (ty, tx) = (t / 16, t mod 16) owning the outputs a = ty + 8 i,
// b' = tx + 16 j.  X is overwritten in place between two barriers a step, and the step's weights
// are read from it directly while the next product begins; odd row pitches keep rows and columns
// free of bank conflicts.  g_{k-1} (or g_{k+1}) comes into registers while step k multiplies.
// (With X in two buffers and the weights turned through a staging buffer, four barriers a step:
// W=32 x L=100, 32 energies 2.42 ms, 2.08 now; W=24 1.25, 1.04.)
constexpr int kNThreads = 128;
constexpr int kNMax = 32;
constexpr size_t kNSmem = sizeof(cf) * (kNMax * (2 * kNMax + 1) + kNMax * (kNMax + 1));

template <int W>
__device__ __forceinline__ void chain_cta_narrow_body(const TaskDesc& d, const TcJob& job,
                                                      const float* __restrict__ eta32,
                                                      const float* __restrict__ phi32,
                                                      const double* __restrict__ gam,
                                                      const cf* __restrict__ gL,
                                                      const cf* __restrict__ gR,
                                                      const cf* __restrict__ start,
                                                      float* __restrict__ weights,
                                                      unsigned char* smem) {
  constexpr int N = 2 * W;                    // the pair's columns
  constexpr int XP = N + 1, GP = W | 1;       // row pitches
  constexpr int RI = (W + 7) / 8;             // output rows a = ty + 8 i
  constexpr int CJ = (N + 15) / 16;           // output columns b' = tx + 16 j
  constexpr int kPre = (W * W + kNThreads - 1) / kNThreads;
  cf* X = reinterpret_cast<cf*>(smem);                     // [c][b']
  cf* Gs = X + W * XP;                                     // [a][c] (-t g_k); Phi at the edges

  const int tid = threadIdx.x;
  const int L = d.L, n = d.n, K = d.K;
  const int dir = job.dir;
  auto m0_of = [&](int yy) { return yy < L ? yy : (yy == L ? 0 : L - 1); };
  const int ys[2] = {job.y0, job.y1};
  const float mt = (float)(-d.t);
  const float* eta = eta32 + d.onsite_off / 2;
  const cf* gsrc = (dir == 0 ? gL : gR) + d.g_off;
  float* wt = weights + d.wt_off;
  auto row_of = [&](int y, int b) -> uint64_t {
    return y < L ? (uint64_t)y * W + b : (uint64_t)n + (uint64_t)(y - L) * W + b;
  };
  auto load_start = [&](int col) {
    const cf* st = start + d.start_off + (uint64_t)ys[col] * W * W;
    for (int i = tid; i < W * W; i += kNThreads) X[(i / W) * XP + col * W + i % W] = st[i];
  };
  // weights of slice k for the columns in `mask`, from X
  auto emit = [&](int k, unsigned mask) {
#pragma unroll
    for (int q = 0; q < (N * W + kNThreads - 1) / kNThreads; ++q) {
      const int i = tid + kNThreads * q;
      const int r = i / W, a = i - r * W;                  // a consecutive: coalesced rows
      const int col = r >= W;
      if (i < N * W && (mask & (1u << col))) {
        const cf v = X[a * XP + r];
        wt[row_of(ys[col], r - col * W) * K + (uint64_t)k * W + a] =
            __fmul_rn(__ldg(eta + k * W + a), __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)));
      }
    }
  };
  // lead weights sum_nu Gamma_nu |(Phi^T X)_nu b'|^2 at a boundary slice: Phi (FP32) takes the g
  // buffer, which no product needs any more (or yet); two threads per column, each half of the
  // modes, then the sum of the halves.  Synchronised before and after.
  auto lead_weights = [&](int k, unsigned mask) {
    float* phis = reinterpret_cast<float*>(Gs);
    float* gams = phis + W * W;
    float* parts = gams + W;
    for (int i = tid; i < W * W; i += kNThreads) phis[i] = phi32[d.phi_off + i];
    for (int i = tid; i < W; i += kNThreads) gams[i] = (float)gam[d.lead_off + i];
    __syncthreads();
    const int r = tid % 64, h = tid / 64;
    if (r < N) {
      float part = 0.f;
      for (int nu = h * (W / 2); nu < (h ? W : W / 2); ++nu) {
        float zr = 0.f, zi = 0.f;
#pragma unroll 8
        for (int a = 0; a < W; ++a) {
          const float p = phis[a * W + nu];
          const cf v = X[a * XP + r];
          zr = __fmaf_rn(p, v.x, zr);
          zi = __fmaf_rn(p, v.y, zi);
        }
        part = __fmaf_rn(gams[nu], __fmaf_rn(zr, zr, __fmul_rn(zi, zi)), part);
      }
      parts[h * N + r] = part;
    }
    __syncthreads();
    if (h == 0 && r < N) {
      const int col = r / W;
      if (mask & (1u << col)) {
        const float lw = parts[r] + parts[N + r];
        const uint64_t base = row_of(ys[col], r - col * W) * K + n;
        if (k == 0) wt[base] = lw;
        if (k == L - 1) wt[base + 1] = lw;
      }
    }
    __syncthreads();
  };

  unsigned have = 0;
  for (int col = 0; col < 2; ++col)
    if (ys[col] >= 0) have |= 1u << col;
  if (dir == 0) {
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
  if (k_first == k_end) return;
  cf gp[kPre];
  auto fetch = [&](int k) {
    const cf* gk = gsrc + (uint64_t)k * W * W;
#pragma unroll
    for (int r = 0; r < kPre; ++r) {
      const int i = tid + kNThreads * r;
      if (i < W * W) gp[r] = gk[i];
    }
  };
  auto put = [&]() {
#pragma unroll
    for (int r = 0; r < kPre; ++r) {
      const int i = tid + kNThreads * r;
      if (i < W * W) Gs[(i / W) * GP + i % W] = cf{mt * gp[r].x, mt * gp[r].y};
    }
  };
  fetch(k_first);
  put();
  const int ty = tid / 16, tx = tid % 16;
  // operand rows and columns; those beyond the block read its last ones and are not stored
  int ra[RI], cb[CJ];
#pragma unroll
  for (int i = 0; i < RI; ++i) ra[i] = (RI * 8 == W ? ty + 8 * i : min(ty + 8 * i, W - 1)) * GP;
#pragma unroll
  for (int j = 0; j < CJ; ++j) cb[j] = CJ * 16 == N ? tx + 16 * j : min(tx + 16 * j, N - 1);
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
#pragma unroll 4
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
          accr[i][j] = fmaf(g[i].x, x[j].x, accr[i][j]);
          accr[i][j] = fmaf(-g[i].y, x[j].y, accr[i][j]);
          acci[i][j] = fmaf(g[i].x, x[j].y, acci[i][j]);
          acci[i][j] = fmaf(g[i].y, x[j].x, acci[i][j]);
        }
    }
    __syncthreads();                                       // X and g have been read
#pragma unroll
    for (int i = 0; i < RI; ++i)
#pragma unroll
      for (int j = 0; j < CJ; ++j) {
        const int a = ty + 8 * i, b = tx + 16 * j;
        if ((RI * 8 == W || a < W) && (CJ * 16 == N || b < N))
          X[a * XP + b] = cf{accr[i][j], acci[i][j]};
      }
    if (more) put();
    __syncthreads();
    emit(k, active);
    if (k == 0 || k == L - 1) lead_weights(k, active);     // the last step of its direction
  }
}

__global__ void __launch_bounds__(kNThreads, 4) chain_cta_narrow_kernel(
    const TaskDesc* __restrict__ tasks, const TcJob* __restrict__ jobs,
    const float* __restrict__ eta32, const float* __restrict__ phi32,
    const double* __restrict__ gam, const cf* __restrict__ gL, const cf* __restrict__ gR,
    const cf* __restrict__ start, float* __restrict__ weights) {
  extern __shared__ __align__(16) unsigned char smem[];
  const TcJob job = jobs[blockIdx.x];
  const TaskDesc d = tasks[job.task];
#define NEGF_CN_CASE(w)                                                                       \
  case w:                                                                                     \
    chain_cta_narrow_body<w>(d, job, eta32, phi32, gam, gL, gR, start, weights, smem);        \
    break;
  switch (d.W) {
    NEGF_CN_CASE(17) NEGF_CN_CASE(18) NEGF_CN_CASE(19) NEGF_CN_CASE(20)
    NEGF_CN_CASE(21) NEGF_CN_CASE(22) NEGF_CN_CASE(23) NEGF_CN_CASE(24)
    NEGF_CN_CASE(25) NEGF_CN_CASE(26) NEGF_CN_CASE(27) NEGF_CN_CASE(28)
    NEGF_CN_CASE(29) NEGF_CN_CASE(30) NEGF_CN_CASE(31) NEGF_CN_CASE(32)
    default: break;
  }
#undef NEGF_CN_CASE
}

}  // namespace

cudaError_t launch_chain_cta(const TaskDesc* d_tasks, const TcJob* d_jobs, uint32_t n_wide,
                             uint32_t n_narrow, uint32_t n_mid, const float* d_eta32,
                             const float* d_phi32, const double* d_gam, const void* d_gL,
                             const void* d_gR, const void* d_start, void* d_weights,
                             uint64_t* d_tab, int32_t* d_err, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  if (n_wide) {
    e = allow_smem(chain_cta_kernel);
    if (e != cudaSuccess) return e;
    chain_cta_kernel<<<n_wide, kThreads, kSmem, s>>>(
        d_tasks, d_jobs, d_eta32, d_phi32, d_gam, static_cast<const cf*>(d_gL),
        static_cast<const cf*>(d_gR), static_cast<const cf*>(d_start),
        static_cast<float*>(d_weights), d_tab, d_err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (n_narrow) {
    e = allow_smem(chain_cta_narrow_kernel);
    if (e != cudaSuccess) return e;
    chain_cta_narrow_kernel<<<n_narrow, kNThreads, kNSmem, s>>>(
        d_tasks, d_jobs + n_wide, d_eta32, d_phi32, d_gam, static_cast<const cf*>(d_gL),
        static_cast<const cf*>(d_gR), static_cast<const cf*>(d_start),
        static_cast<float*>(d_weights));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return launch_chain_mid(d_tasks, d_jobs + n_wide + n_narrow, n_mid, d_eta32, d_phi32, d_gam,
                          d_gL, d_gR, d_start, d_weights, s);
}

}  // namespace negf
