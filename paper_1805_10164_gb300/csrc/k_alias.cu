// Alias-table construction for the Step 6' categorical draw.
//
// Sec. III.B draws the next index by a cumulative sum and a search (O(K) per step).  The walk
// here uses Walker's alias method (one table entry per draw), so each row of weights is turned
// into K slots (threshold, alias).  One warp builds one row, in exact integer arithmetic on a
// quantised copy of the row, by a parallel "sweep" construction (in the spirit of
// Hubschle-Schneider and Sanders, "Parallel weighted random sampling", ESA 2019), written from
// this derivation:
//
//   Quantise: scale the row by a power of two so that its largest weight lies in [2^31, 2^32)
//   and truncate to integers m_i (exact scaling, no rounding of the others beyond 2^-32 of the
//   largest); T = sum m_i is exact.  Then u_i = floor(m_i K 2^32 / T) (by a 64 x 64 -> 128-bit
//   product with a per-row reciprocal), and the integer remainder K 2^32 - sum(u) goes to the
//   largest item, so that sum(u) = K 2^32 exactly and every slot holds exactly 2^32 units.  Light items (u < 2^32) in index order carry deficits 2^32 - u with
//   inclusive prefix sums Lc_r; heavy items (u >= 2^32) carry excesses u - 2^32 with inclusive
//   prefix sums Ec_j.  Heavy j owns the interval [Ec_{j-1}, Ec_j) of the deficit line.
//   * light r keeps thr = u and aliases the heavy whose interval contains its start Lc_{r-1};
//   * heavy j (not the last) is consumed past its excess by the light interval (Lc_{r-1}, Lc_r]
//     that contains Ec_j; its slot keeps thr = 2^32 - (Lc_r - Ec_j) and aliases heavy j+1.
//     If no light interval contains Ec_j (Ec_j == 0) the slot is full;
//   * the last heavy is full (sum of deficits == sum of excesses exactly).
//   Every item then holds exactly u_i of the K 2^32 units.
// Full slots store thr = 2^32 - 1 and alias = self.  The FP64 row sum is also the sum-rule check
// of Sec. II.D (each row must add up to <i|A|i>, which the diagonal-block kernel stored).
#include <cuda_runtime.h>
#include <math.h>

#include "alias_small.cuh"
#include "level2.cuh"
#include "negf_internal.cuh"

namespace negf {
namespace {

constexpr uint64_t kSlot = 1ull << 32;

__device__ __forceinline__ uint64_t pack(uint32_t thr, uint32_t alias) {
  return (uint64_t)thr | ((uint64_t)alias << 32);
}

// What bounds it: instructions, on few warps per SM (shared memory per warp).  A row passes
// through its items three times to form the units (largest weight; integer weights and their
// total; units and their sums), once to list lights and heavies, and once, over the list of
// lights, to write the slots: a light's own, and those of the heavies whose excess ends within
// its interval, so that no slot needs a search.  Measured, GB300, against six passes with a
// search per slot: rows of 502 slots (W=10 x L=50, 64 energies) 0.300 -> 0.218 ms, of 1602
// (W=16 x L=100, 16 energies, weights kept) 1.38 -> 0.65, of 2002 (W=40 x L=50, 16 tasks)
// 2.03 -> 1.35, FP64 rows of 502 0.61 -> 0.54.
//
// A row of more than kAliasWarpRow slots is built by four warps, shorter ones by one: a row's
// arrays (22 bytes a slot) leave room for few rows per SM, and one warp each then leaves it
// idle between its dependent steps; four warps share a row's arrays for seven barriers a row.
// One warp against four, ms: 702 slots (64 energies) 0.39, 0.78; 1002 (64,128 rows) 0.91, 1.01;
// 1602 0.65, 0.56; 1702 (32 energies) 1.98, 1.25; 2002 (16 tasks) 1.34, 0.83.  A build launches
// one kernel per class of row lengths among its tasks, the short rows (up to kAliasShortRow) with
// shared memory for their own length: 1280 uneven tasks 42 -> 30 ms.
//
// Each of the group's threads (the lanes of its NW warps) owns a block of npl consecutive items,
// npl = ceil(K / (32 NW)).  Per-item values live in shared memory at slot
// (i / npl) * pitch + i % npl, with an odd pitch (npl or npl + 1) so that the lanes walking their
// blocks in step touch 32 different banks.
constexpr int kAliasShortRow = 512, kAliasWarpRow = 1200;
template <int NW>
__host__ __device__ inline int alias_npl(int K) { return (K + 32 * NW - 1) / (32 * NW); }
template <int NW>
__host__ __device__ inline int alias_pitch(int K) { return alias_npl<NW>(K) | 1; }
// Per-group shared memory: s_u, s_c : u64 [32 NW pitch] | the row's weights (32 NW pitch elements
// of `elem` bytes, or those of 64 FP64 mode weights) | s_x : u16 [cap] | exchange between warps
template <int NW>
__host__ __device__ inline size_t alias_stage_bytes(int cap, int elem) {
  const size_t row = (size_t)32 * NW * alias_pitch<NW>(cap) * elem;
  const size_t modes = (size_t)32 * NW * alias_pitch<NW>(64) * sizeof(double);
  return ((row > modes ? row : modes) + 15) & ~(size_t)15;
}
struct AliasExchange {            // one slot per warp of the group
  uint64_t a, b, c;
  uint32_t m, k;
};
template <int NW>
__host__ __device__ inline size_t alias_group_bytes(int cap, int elem) {
  const size_t slots = (size_t)32 * NW * alias_pitch<NW>(cap);
  return 2 * slots * sizeof(uint64_t) + alias_stage_bytes<NW>(cap, elem) +
         (((size_t)cap * sizeof(uint16_t) + 15) & ~(size_t)15) +
         (NW > 1 ? 2 * NW * sizeof(AliasExchange) : 0);
}
// A group's arrays in its shared memory, and its threads
template <int NW>
struct AliasGroup {
  uint64_t *u, *c;
  unsigned char* stage;
  uint16_t* x;
  AliasExchange* ex;              // two sets in turn
  int lane, t;                    // lane of the warp, thread of the group
  int bar;                        // the group's barrier
  __device__ AliasGroup(unsigned char* smem, int group, int cap, int elem) {
    unsigned char* base = smem + (size_t)group * alias_group_bytes<NW>(cap, elem);
    u = reinterpret_cast<uint64_t*>(base);
    c = u + (size_t)32 * NW * alias_pitch<NW>(cap);
    stage = reinterpret_cast<unsigned char*>(c + (size_t)32 * NW * alias_pitch<NW>(cap));
    unsigned char* xb = stage + alias_stage_bytes<NW>(cap, elem);
    x = reinterpret_cast<uint16_t*>(xb);
    ex = reinterpret_cast<AliasExchange*>(xb + (((size_t)cap * sizeof(uint16_t) + 15) & ~(size_t)15));
    lane = threadIdx.x & 31;
    t = threadIdx.x % (32 * NW);
    bar = 1 + group;
  }
  __device__ void sync() const {
    if (NW == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(bar), "n"(32 * NW) : "memory");
  }
};

// f(i, slot) for the thread's items i = t, t + 32 NW, ... of a K-item row
template <int NW, typename F>
__device__ __forceinline__ void alias_strided(const AliasGroup<NW>& g, int K, F f) {
  constexpr int NT = 32 * NW;
  const int npl = alias_npl<NW>(K), pitch = alias_pitch<NW>(K);
  const int q32 = NT / npl, r32 = NT - q32 * npl;
  int q = g.t / npl, r = g.t - q * npl;
  for (int i = g.t; i < K; i += NT) {
    f(i, q * pitch + r);
    q += q32;
    r += r32;
    if (r >= npl) { r -= npl; ++q; }
  }
}

// Asynchronous global -> shared copies of 4 or 8 bytes (the weights of the next row).
template <int kBytes>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(kBytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t fixp(float w, int sh) { return small_fixp(w, sh); }
__device__ __forceinline__ uint32_t fixp(double w, int sh) { return __double2uint_rz(ldexp(w, sh)); }

// Build one row by the group's threads.  sm.stage: the K weights, item i at its slot (alias_strided); A: the value the
// row must sum to (checked when check_A, to tol A + atol: a row whose spectral weight is at the
// rounding level of G, such as an orbital no open channel reaches, carries only rounding noise);
// out: K entries; rowsum_out: receives the row sum.  after_stage() is called by every lane once
// the weights have been read (the caller reuses the stage for the next row).
template <typename R, int NW, typename After>
__device__ void alias_row(const AliasGroup<NW>& sm, int K, double A, bool check_A, double tol,
                          double atol, uint64_t* __restrict__ out, double* rowsum_out,
                          int32_t* err, After after_stage) {
  constexpr int NT = 32 * NW;
  const int lane = sm.lane, warp = sm.t >> 5;
  const unsigned FULL = 0xffffffffu;
  const int npl = alias_npl<NW>(K), pitch = alias_pitch<NW>(K);
  const int i0 = min(K, sm.t * npl);                            // this thread's items [i0, i1)
  const int i1 = min(K, i0 + npl);
  const int mine = i1 - i0;
  uint64_t* my_u = sm.u + sm.t * pitch;
  const R* w = reinterpret_cast<const R*>(sm.stage);
  const R* my_w = w + sm.t * pitch;
  AliasExchange* const ex = sm.ex;
  // pass 1: largest weight; FP64 rows also take their FP64 sum here (lane-strided order, tree to
  // lane 0)
  R wmax = 0;
  bool bad = false;
  for (int k = 0; k < mine; ++k) {
    const R v = my_w[k];
    const bool ok = v >= 0 && v < (R)INFINITY;
    bad |= !ok;
    if (ok && v > wmax) wmax = v;
  }
  double part = 0.0;
  if (sizeof(R) == 8 && warp == 0)                // (by one warp, whatever NW is: one order)
    for (int i = lane; i < K; i += 32) part += (double)w[i / npl * pitch + i % npl];
  for (int off = 16; off > 0; off >>= 1) wmax = max(wmax, __shfl_xor_sync(FULL, wmax, off));
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(err, ERR_NONFINITE);
  if (NW > 1) {
    R* wm = reinterpret_cast<R*>(&ex[warp].a);
    if (lane == 0) *wm = wmax;
    sm.sync();
#pragma unroll
    for (int v = 0; v < NW; ++v) wmax = max(wmax, *reinterpret_cast<const R*>(&ex[v].a));
  }
  if (!(wmax > 0)) {
    sm.sync();
    after_stage();
    if (sm.t == 0) *rowsum_out = 0.0;
    if (sm.t == 0 && check_A && A > 1e-300 && A > atol) atomicOr(err, ERR_ROWSUM);
    for (int i = sm.t; i < K; i += NT) out[i] = pack(0xffffffffu, (uint32_t)i);
    return;
  }
  int e2p = 0;
  if (sizeof(R) == 4) frexpf((float)wmax, &e2p);  // wmax = f 2^e2p, f in [0.5, 1)
  else frexp((double)wmax, &e2p);
  const int sh = 32 - e2p;                          // wmax 2^sh in [2^31, 2^32)
  auto unit = [&](int k) {
    const R v = my_w[k];
    return v > 0 && v < (R)INFINITY ? fixp(v, sh) : 0u;
  };
  // pass 2: integer weights m_i, T = sum m_i, and the first index of the largest
  uint64_t T = 0;
  uint32_t mmax = 0;
  int imax = 0x7fffffff;
  for (int k = 0; k < mine; ++k) {
    const uint32_t m = unit(k);
    if (sizeof(R) == 8) my_u[k] = m;
    T += m;
    if (m > mmax) { mmax = m; imax = i0 + k; }
  }
  for (int off = 16; off > 0; off >>= 1) {
    T += __shfl_xor_sync(FULL, T, off);
    const uint32_t om = __shfl_xor_sync(FULL, mmax, off);
    const int oi = __shfl_xor_sync(FULL, imax, off);
    if (om > mmax || (om == mmax && oi < imax)) { mmax = om; imax = oi; }
  }
  if (NW > 1) {
    AliasExchange* const e2 = ex + NW;
    if (lane == 0) {
      e2[warp].a = T;
      e2[warp].m = mmax;
      e2[warp].k = (uint32_t)imax;
    }
    sm.sync();
    T = 0;
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      T += e2[v].a;
      if (e2[v].m > mmax || (e2[v].m == mmax && (int)e2[v].k < imax)) {
        mmax = e2[v].m;
        imax = (int)e2[v].k;
      }
    }
  }
  // row sum: FP64 weights are summed in FP64; FP32 weights use the exact fixed-point sum
  // (within K 2^-32 of the largest weight)
  if (sizeof(R) == 8)
    for (int off = 16; off > 0; off >>= 1) part += __shfl_down_sync(FULL, part, off);
  // the FP64 steps run on one lane of a warp only (FP64 throughput is low); the reciprocal is
  // broadcast
  uint64_t rcp = 0;
  if (lane == 0) {
    const double total = sizeof(R) == 8 ? part : ldexp((double)T, -sh);
    rcp = (uint64_t)(ldexp(1.0, 94) / (double)T);   // < 2^63 since T >= 2^31
    if (sm.t == 0) *rowsum_out = total;
    if (sm.t == 0 && check_A && A > 1e-300 && fabs(total - A) > tol * A + atol) atomicOr(err, ERR_ROWSUM);
  }
  rcp = __shfl_sync(FULL, rcp, 0);
  // pass 3: u_i = floor(m_i K 2^32 / T) = (m_i K) (2^94 / T) / 2^62, a 48 x 63-bit product in
  // 32-bit limbs.  m_i <= T, so no unit count exceeds K 2^32; K 2^32 / T > 1 + 2^-33 exceeds the
  // reciprocal's error, so u_i grows strictly with m_i and the largest m has the largest u.
  // Lights (u < 2^32) carry deficits 2^32 - u, heavies excesses u - 2^32.
  const uint32_t r0 = (uint32_t)rcp, r1 = (uint32_t)(rcp >> 32);
  uint64_t usum = 0, dl = 0;
  uint32_t cnt = 0;                               // lights | heavies << 16
  for (int k = 0; k < mine; ++k) {
    const uint32_t m = sizeof(R) == 8 ? (uint32_t)my_u[k] : unit(k);
    const uint64_t q = (uint64_t)m * (uint32_t)K;
    const uint32_t q0 = (uint32_t)q, q1 = (uint32_t)(q >> 32);
    const uint64_t p = (uint64_t)q0 * r1 + (((uint64_t)q0 * r0) >> 32);
    const uint64_t s = (uint64_t)q1 * r0 + (uint32_t)p;
    const uint64_t hi = (uint64_t)q1 * r1 + (p >> 32) + (s >> 32);
    const uint64_t u = (hi << 2) | ((uint32_t)s >> 30);
    my_u[k] = u;
    usum += u;
    const bool heavy = u >= kSlot;
    cnt += heavy ? 1u << 16 : 1u;
    dl += heavy ? 0u : (uint32_t)u;               // lights' units
  }
  // the other exchange set has been read by every warp (each has passed the barrier after it)
  if (NW > 1) {
    uint64_t s = usum;
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(FULL, s, off);
    if (lane == 0) ex[warp].b = s;
  }
  sm.sync();
  after_stage();
  const int nl_mine = (int)(cnt & 0xffffu), nh_mine = (int)(cnt >> 16);
  uint64_t dh = usum - dl - ((uint64_t)nh_mine << 32);          // excesses
  dl = ((uint64_t)nl_mine << 32) - dl;                            // deficits
  if (NW == 1) {
    for (int off = 16; off > 0; off >>= 1) usum += __shfl_xor_sync(FULL, usum, off);
  } else {
    usum = 0;
#pragma unroll
    for (int v = 0; v < NW; ++v) usum += ex[v].b;
  }
  if (i0 <= imax && imax < i1) {                  // the signed remainder goes to the largest item
    const uint64_t rem = ((uint64_t)K << 32) - usum;
    const uint64_t u0 = my_u[imax - i0], u1 = u0 + rem;
    my_u[imax - i0] = u1;
    if (u0 >= kSlot) {
      dh += rem;
    } else if (u1 >= kSlot) {
      cnt += (1u << 16) - 1u;
      dl -= kSlot - u0;
      dh += u1 - kSlot;
    } else {
      dl -= rem;
    }
  }
  // exclusive prefix over the lanes of counts and sums
  uint32_t cx = cnt;
  uint64_t lx = dl, hx = dh;                      // inclusive scans
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t oc = __shfl_up_sync(FULL, cx, off);
    const uint64_t ol = __shfl_up_sync(FULL, lx, off);
    const uint64_t oh = __shfl_up_sync(FULL, hx, off);
    if (lane >= off) { cx += oc; lx += ol; hx += oh; }
  }
  uint32_t ctot = __shfl_sync(FULL, cx, 31);
  if (NW > 1) {
    AliasExchange* const e2 = ex + NW;
    if (lane == 31) {
      e2[warp].a = lx;
      e2[warp].b = hx;
      e2[warp].m = cx;
    }
    sm.sync();
    ctot = 0;
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      ctot += e2[v].m;
      if (v < warp) {
        cx += e2[v].m;
        lx += e2[v].a;
        hx += e2[v].b;
      }
    }
  }
  const int nl = (int)(ctot & 0xffffu), nh = (int)(ctot >> 16);
  int r = (int)((cx - cnt) & 0xffffu), j = (int)((cx - cnt) >> 16);   // first light / heavy
  uint64_t runl = lx - dl, runh = hx - dh;                             // of this lane
  // pass 4: Lc_r (inclusive deficit prefix, light order) from the front of s_c, Ec_j (inclusive
  // excess prefix, heavy order) from the back; s_x holds the item index of each
  for (int k = 0; k < mine; ++k) {
    const uint64_t u = my_u[k];
    const bool heavy = u >= kSlot;
    if (heavy) runh += u - kSlot;
    else runl += kSlot - u;
    const int at = heavy ? K - 1 - j : r;
    sm.c[at] = heavy ? runh : runl;
    sm.x[at] = (uint16_t)(i0 + k);
    j += heavy;
    r += !heavy;
  }
  sm.sync();
  if (nl == 0 || nh == 0) {   // every item holds one slot (nh == 0 cannot happen: the sum is K 2^32)
    for (int i = sm.t; i < K; i += NT) out[i] = pack(0xffffffffu, (uint32_t)i);
    return;
  }
  auto Ec = [&](int jj) { return sm.c[K - 1 - jj]; };
  auto Xh = [&](int jj) { return (uint32_t)sm.x[K - 1 - jj]; };
  auto Lc = [&](int rr) { return sm.c[rr]; };
  // pass 5: entries, into s_u by item index (s_u is dead from here).  The lanes split the list of
  // lights into contiguous ranges.  Light r (start Lc_{r-1}, u_r = 2^32 - (Lc_r - Lc_{r-1}))
  // aliases heavy j, the first whose excess interval [Ec_{j-1}, Ec_j) reaches past its start;
  // the heavies (but the last) that end within (Lc_{r-1}, Lc_r] are consumed past their excess
  // by this light: heavy j keeps 2^32 - (Lc_r - Ec_j) and aliases heavy j + 1.  Heavies without
  // excess at the front of the list (Ec = 0) and the last heavy are full.
  {
    const int ra = sm.t * nl / NT, rb = (sm.t + 1) * nl / NT;
    if (ra < rb) {
      uint64_t st = ra == 0 ? 0ull : Lc(ra - 1);
      int jc = 0, hi = nh - 1;                            // first j with Ec_j > st, or the last
      while (jc < hi) {
        const int mid = (jc + hi) >> 1;
        if (Ec(mid) > st) hi = mid; else jc = mid + 1;
      }
      if (ra == 0)
        for (int jj = 0; jj < jc; ++jj) sm.u[Xh(jj)] = pack(0xffffffffu, Xh(jj));
      uint64_t Ej = Ec(jc);
      uint32_t xj = Xh(jc);
      for (int rr = ra; rr < rb; ++rr) {
        const uint64_t Lr = Lc(rr);
        sm.u[sm.x[rr]] = pack((uint32_t)(st - Lr), xj);    // 2^32 - (Lr - st)
        while (jc < nh - 1 && Ej <= Lr) {
          const uint32_t xn = Xh(jc + 1);
          const uint64_t used = Lr - Ej;                   // consumed beyond the excess, <= 2^32
          sm.u[xj] = used > 0 ? pack((uint32_t)(kSlot - used), xn) : pack(0xffffffffu, xj);
          ++jc;
          Ej = Ec(jc);
          xj = xn;
        }
        st = Lr;
      }
    }
    if (sm.t == 0) sm.u[Xh(nh - 1)] = pack(0xffffffffu, Xh(nh - 1));
  }
  sm.sync();
  for (int i = sm.t; i < K; i += NT) out[i] = sm.u[i];
  sm.sync();
}

// Rows of the tasks with min_K < K <= max_K, a row per group of NW warps.
template <typename R, int NW>
__global__ void alias_kernel(const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t total_jobs,
                             int min_K, int max_K, int cap, double tol,
                             const R* __restrict__ weights, double* __restrict__ rowsum,
                             const double* __restrict__ mode_w, uint64_t* __restrict__ tab,
                             uint64_t* __restrict__ mode_tab, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int group = threadIdx.x / (32 * NW), ngroups = blockDim.x / (32 * NW);
  const AliasGroup<NW> sm(smem_raw, group, cap, (int)sizeof(R));
  const uint32_t stride = gridDim.x * ngroups;
  // The group's first job at or after jb whose task is of this class, and that task: jobs of a
  // group only increase, so the search starts at the last task found and passes over the tasks
  // of the other class.
  auto next_job = [&](uint32_t jb, int& task) -> uint32_t {
    int lo = task, hi = n_tasks - 1;
    while (lo < hi && jb < total_jobs) {
      const int mid = (lo + hi + 1) >> 1;
      if (tasks[mid].row_base <= jb) lo = mid; else hi = mid - 1;
    }
    while (jb < total_jobs) {
      const int K = tasks[lo].K;
      if (K > min_K && K <= max_K) break;
      if (lo + 1 >= n_tasks) return total_jobs;
      const uint32_t base = tasks[++lo].row_base;
      if (base > jb) jb += (base - jb + stride - 1) / stride * stride;
      while (lo + 1 < n_tasks && tasks[lo + 1].row_base <= jb) ++lo;
    }
    task = lo;
    return jb < total_jobs ? jb : total_jobs;
  };
  // the weights of job jb go to the stage by asynchronous copies (one commit group)
  auto stage = [&](uint32_t jb, int task) {
    const TaskDesc& d = tasks[task];
    const int row = (int)(jb - d.row_base);
    if (row < d.rows) {
      const R* src = weights + d.wt_off + (uint64_t)row * d.K;
      R* dst = reinterpret_cast<R*>(sm.stage);
      alias_strided<NW>(sm, d.K, [&](int i, int slot) { cp_async<(int)sizeof(R)>(dst + slot, src + i); });
    } else {
      const double* src = mode_w + d.mode_off + (row - d.rows) * d.W;
      double* dst = reinterpret_cast<double*>(sm.stage);
      alias_strided<NW>(sm, d.W, [&](int i, int slot) { cp_async<8>(dst + slot, src + i); });
    }
    cp_async_commit();
  };
  int task = 0;
  uint32_t job = next_job(blockIdx.x * ngroups + group, task);
  if (job < total_jobs) stage(job, task);
  while (job < total_jobs) {
    const TaskDesc& d = tasks[task];
    const int row = (int)(job - d.row_base);
    const double A = rowsum[job];                 // <i|A|i> (rows) or c_p (mode rows)
    int task2 = task;
    const uint32_t next = total_jobs - job > stride ? next_job(job + stride, task2) : total_jobs;
    auto after = [&]() {
      if (next < total_jobs) stage(next, task2);
    };
    cp_async_wait_all();
    sm.sync();
    if (row < d.rows) {
      alias_row<R, NW>(sm, d.K, A, true, tol, 1e-13 / d.t, tab + d.tab_off + (uint64_t)row * d.K,
                       rowsum + job, err, after);
    } else {
      const int p = row - d.rows;
      alias_row<double, NW>(sm, d.W, A, true, 1e-9, 1e-13 / d.t, mode_tab + d.mode_off + p * d.W,
                            rowsum + job, err, after);
    }
    sm.sync();
    job = next;
    task = task2;
  }
  cp_async_wait_all();
}

// ---- Level-2 inverse-CDF blocks of two-level tables --------------------------------------
//
// Within a slice the site is drawn by the paper's own categorical draw (Sec. III.B: cumulative
// sum of the weights, normalised, the first entry above a uniform), in integers: for the W site
// weights w_a of (table row, slice), c_a = floor(2^31 P_a / S) with P_a = sum_{b <= a} w_b and
// S = P_{W-1}, for a < W - 1; c_{W-1} and the padding of the last octet are 2^31.  Octet g holds
// c_{8g .. 8g+7}; for W > 8 an 8-word guide precedes the octets, guide_g = c_{8g+7} for
// g < G - 1 and 2^31 after (G = ceil(W / 8)).  The walk draws v = x >> 1 (31 bits), takes
// g = #{guide words <= v} and the site 8g + #{words of octet g <= v}, so site a has probability
// (c_a - c_{a-1}) / 2^31 and a zero weight is never drawn.  A slice whose weights sum to zero
// gets 2^31 everywhere (its level-1 weight is zero, so it is never drawn).
// FP32 weights: s = 2^sh with (FP32 sum) s in [2^29, 2^30); m_a = floor(w_a s) (exact scaling
// and truncation), P_a = sum m (exact integers, < 2^31), T = P_{W-1}, c_a = floor(P_a R / 2^31)
// with R = floor(2^62 / T) (within one unit below floor(2^31 P_a / T), nondecreasing in P_a),
// c_a = 2^31 where P_a = T; the slice's level-1 weight is T / s.  FP64 weights: P_a, S and c_a
// in FP64, level-1 weight S.
// One warp per table row, chunks of 32 slices: the chunk's weights are staged by coalesced loads,
// each lane forms one slice's block in registers and writes it into its shared region (odd pitch
// in 4-byte words), and the chunk's blocks (32 consecutive blocks of the row) leave by coalesced
// stores.
constexpr int kL2Warps = 4;

// Region pitch in 4-byte words: holds W weights of type R and a block of B2 words; odd for
// 4-byte accesses, 2 mod 4 for 8-byte ones (conflict-free across a half-warp).
template <typename R>
__host__ __device__ inline int level2_pitch(int W, int B2) {
  const int need = (int)(W * sizeof(R) / 4) > B2 ? (int)(W * sizeof(R) / 4) : B2;
  if (sizeof(R) == 4) return need | 1;
  int p = (need + 1) & ~1;
  if ((p & 3) == 0) p += 2;
  return p;
}

template <typename R, int WB>
__device__ __forceinline__ bool level2_block(uint32_t* reg, int W, int B2, R* total) {
  const R* wk = reinterpret_cast<const R*>(reg);
  uint32_t c[WB];
  bool ok = true;
  R tot = 0;
  if constexpr (sizeof(R) == 4) {
    float t32 = 0.f;
    ok = level2_fp32<WB>([&](int a) { return wk[a]; }, W, c, &t32);
    tot = t32;
  } else {
    double S = 0.0;
#pragma unroll
    for (int a = 0; a < WB; ++a)
      if (a < W) S += wk[a];
    if (!(S >= 0.0 && S < INFINITY)) ok = false;
    if (S > 0.0 && S < INFINITY) {
      const double scale = 2147483648.0 / S;
      double P = 0.0;
#pragma unroll
      for (int a = 0; a < WB; ++a) {
        P += a < W ? wk[a] : 0.0;
        c[a] = P >= S ? kCdfOne : min(__double2uint_rz(P * scale), kCdfOne - 1u);
      }
      tot = S;
    } else {
#pragma unroll
      for (int a = 0; a < WB; ++a) c[a] = kCdfOne;
    }
  }
  // c_{W-1} and the padding of the last octet are 2^31 (the weights have been read)
  const int G = (W + 7) >> 3;
  uint32_t* oct = G > 1 ? reg + 8 : reg;
#pragma unroll
  for (int a = 0; a < WB; ++a)
    if (a < 8 * G) oct[a] = a < W - 1 ? c[a] : kCdfOne;
  if (G > 1) {
#pragma unroll
    for (int g = 0; g < 8; ++g) reg[g] = (g < G - 1 && 8 * g + 7 < WB) ? c[8 * g + 7] : kCdfOne;
  }
  *total = tot;
  return ok;
}

template <typename R, int WB>
__global__ void __launch_bounds__(32 * kL2Warps) level2_cdf_kernel(
    const TaskDesc* __restrict__ tasks, int n_tasks, uint32_t n_jobs, R* __restrict__ weights,
    uint64_t* __restrict__ tab, int32_t* err) {
  extern __shared__ __align__(16) unsigned char l2_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t job = blockIdx.x * kL2Warps + warp;
  if (job >= n_jobs) return;
  int lo = 0, hi = n_tasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].row_base <= job) lo = mid; else hi = mid - 1;
  }
  const TaskDesc& d = tasks[lo];
  if (d.layout != NEGF_LAYOUT_TWO_LEVEL || d.l2_fused) return;   // fused: written by the chain
  const int row = (int)(job - d.row_base);
  if (row >= d.rows) return;
  const int W = d.W, L = d.L, n = d.n;
  const int B2 = level2_words(W);
  const int PW = level2_pitch<R>(W, B2);
  uint32_t* wbase = reinterpret_cast<uint32_t*>(l2_smem) + (size_t)warp * 32 * PW;
  const R* wr = weights + d.wt_off + (uint64_t)row * d.K;
  R* l1 = weights + d.l1w_off + (uint64_t)row * (L + 2);
  uint32_t* l2 = reinterpret_cast<uint32_t*>(tab + d.tab_off) + (uint64_t)row * L * B2;
  constexpr int EW = (int)(sizeof(R) / 4);          // words per weight
  const int eq = 32 / W, er = 32 - (32 / W) * W;
  bool ok = true;
  for (int k0 = 0; k0 < L; k0 += 32) {
    const int ns = min(32, L - k0);
    const R* wc = wr + (uint64_t)k0 * W;
    if (EW == 1 && (W & 1) == 0 && (reinterpret_cast<uintptr_t>(wc) & 7) == 0) {
      // FP32 pairs (a pair never straddles two slices when W is even)
      const int hw = W >> 1;
      const int pq = 32 / hw, pr = 32 - (32 / hw) * hw;
      int q = lane / hw, r = lane - q * hw;
      for (int p = lane; p < ns * hw; p += 32) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(wc) + p);
        float* dst = reinterpret_cast<float*>(wbase + q * PW) + 2 * r;
        dst[0] = v.x;
        dst[1] = v.y;
        q += pq;
        r += pr;
        if (r >= hw) { r -= hw; ++q; }
      }
    } else {
      int q = lane / W, r = lane - q * W;
      for (int i = lane; i < ns * W; i += 32) {
        reinterpret_cast<R*>(wbase + q * PW)[r] = wc[i];
        q += eq;
        r += er;
        if (r >= W) { r -= W; ++q; }
      }
    }
    __syncwarp();
    if (lane < ns) {
      R tot = 0;
      ok &= level2_block<R, WB>(wbase + lane * PW, W, B2, &tot);
      l1[k0 + lane] = tot;
    }
    __syncwarp();
    // the chunk's ns blocks are contiguous; blocks are multiples of 8 words, the row's level 2
    // starts 32-byte aligned, so four consecutive words of one block leave as one 16-byte store
    uint32_t* oc = l2 + (uint64_t)k0 * B2;
    {
      int q = (4 * lane) / B2, r = 4 * lane - q * B2;
      const int sq = 128 / B2, sr = 128 - (128 / B2) * B2;
      for (int i = 4 * lane; i < ns * B2; i += 128) {
        const uint32_t* src = wbase + q * PW + r;
        *reinterpret_cast<uint4*>(oc + i) = make_uint4(src[0], src[1], src[2], src[3]);
        q += sq;
        r += sr;
        while (r >= B2) { r -= B2; ++q; }
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    l1[L] = wr[n];
    l1[L + 1] = wr[n + 1];
  }
  if (__any_sync(0xffffffffu, !ok) && lane == 0) atomicOr(err, ERR_NONFINITE);
}

// Step 7' energy rows of inelastic Buttiker probes (Sec. II.F, Eq. draw_E_last): for task t (the
// energy E_e of its wire) and site i, the alias row over the wire's grid energies e' of
//   w_e' K(E_e' - E_e) A_ii(E_e'),   K(dE) = exp(-dE^2 / (2 sigma^2)) (the identity for
// sigma = 0), A_ii(E_e') the row sum of site row i of the wire's task at e' (after the alias
// build), w_e' the energy's quadrature weight.  One warp per (task, site) row, into
// etab + eoff(t) + i nE.
__global__ void energy_alias_kernel(const TaskDesc* __restrict__ tasks, int n_tasks,
                                    const EnergyDesc* __restrict__ edesc,
                                    const uint32_t* __restrict__ job_base, uint32_t total_jobs,
                                    int cap, double sigma, const double* __restrict__ rowsum,
                                    uint64_t* __restrict__ etab, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const AliasGroup<1> sm(smem_raw, warp, cap, (int)sizeof(double));
  double* s_w = reinterpret_cast<double*>(sm.stage);
  for (uint32_t job = blockIdx.x * nwarps + warp; job < total_jobs; job += gridDim.x * nwarps) {
    int lo = 0, hi = n_tasks - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (job_base[mid] <= job) lo = mid; else hi = mid - 1;
    }
    const TaskDesc& d = tasks[lo];
    const EnergyDesc ed = edesc[lo];
    const int i = (int)(job - job_base[lo]);
    const int nE = ed.nE;
    const double inv2s2 = sigma > 0.0 ? 0.5 / (sigma * sigma) : 0.0;
    alias_strided<1>(sm, nE, [&](int ep, int slot) {
      const TaskDesc& dp = tasks[ed.t0 + ep];
      const double dE = dp.E - d.E;
      const double K = sigma > 0.0 ? exp(-dE * dE * inv2s2) : (ep == d.e_idx ? 1.0 : 0.0);
      s_w[slot] = dp.w_E * K * rowsum[dp.row_base + i];
    });
    __syncwarp();
    double total = 0.0;
    alias_row<double, 1>(sm, nE, 0.0, false, 0.0, 0.0, etab + ed.eoff + (uint64_t)i * nE, &total,
                      err, [] {});
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_two_level_split(const TaskDesc* d_tasks, int n_tasks, uint32_t n_jobs,
                                   int precision, void* d_weights, uint64_t* d_tab,
                                   int32_t* d_err, cudaStream_t s, int max_W) {
  if (n_jobs == 0 || n_tasks == 0) return cudaSuccess;
  const unsigned blocks = (n_jobs + kL2Warps - 1) / kL2Warps;
  auto run = [&](auto kernel, auto tag, int wb) -> cudaError_t {
    using R = decltype(tag);
    // shared memory for the widest slice the kernel instance takes (W <= wb)
    int pw = 0;
    for (int W = 1; W <= wb; ++W) {
      const int p = level2_pitch<R>(W, level2_words(W));
      pw = p > pw ? p : pw;
    }
    const size_t smem = (size_t)kL2Warps * 32 * pw * 4;
    const cudaError_t e = allow_smem(kernel);
    if (e != cudaSuccess) return e;
    kernel<<<blocks, 32 * kL2Warps, smem, s>>>(d_tasks, n_tasks, n_jobs, static_cast<R*>(d_weights),
                                               d_tab, d_err);
    return cudaGetLastError();
  };
  if (precision == NEGF_FP64) {
    if (max_W <= 16) return run(level2_cdf_kernel<double, 16>, 0.0, 16);
    if (max_W <= 32) return run(level2_cdf_kernel<double, 32>, 0.0, 32);
    return run(level2_cdf_kernel<double, 64>, 0.0, 64);
  }
  if (max_W <= 16) return run(level2_cdf_kernel<float, 16>, 0.f, 16);
  if (max_W <= 32) return run(level2_cdf_kernel<float, 32>, 0.f, 32);
  return run(level2_cdf_kernel<float, 64>, 0.f, 64);
}

cudaError_t launch_energy_tables(const TaskDesc* d_tasks, int n_tasks, const EnergyDesc* d_edesc,
                                 const uint32_t* d_job_base, uint32_t total_jobs, int max_nE,
                                 double sigma, const double* d_rowsum, uint64_t* d_etab,
                                 int32_t* d_err, cudaStream_t s) {
  if (total_jobs == 0) return cudaSuccess;
  const int cap = max_nE < 64 ? 64 : max_nE;
  const size_t per_warp = alias_group_bytes<1>(cap, (int)sizeof(double));
  int warps = 4;
  while (warps > 1 && per_warp * warps > 200 * 1024) --warps;
  const size_t smem = per_warp * warps;
  if (smem > 220 * 1024) return cudaErrorInvalidValue;     // energy grids beyond shared memory
  const cudaError_t e = allow_smem(energy_alias_kernel);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  uint32_t blocks = (total_jobs + warps - 1) / warps;
  if (blocks > (uint32_t)sms * 16) blocks = (uint32_t)sms * 16;
  energy_alias_kernel<<<blocks, warps * 32, smem, s>>>(d_tasks, n_tasks, d_edesc, d_job_base,
                                                      total_jobs, cap, sigma, d_rowsum, d_etab,
                                                      d_err);
  return cudaGetLastError();
}

int alias_warps_max(int max_K) {
  const int cap = max_K < 64 ? 64 : max_K < kAliasWarpRow ? max_K : kAliasWarpRow;
  const size_t per_warp = alias_group_bytes<1>(cap, (int)sizeof(double));
  int w = 16;
  while (w > 1 && per_warp * w > 200 * 1024) --w;
  return w;
}

namespace {
template <typename R, int NW>
cudaError_t alias_class(const TaskDesc* d_tasks, int n_tasks, uint32_t total_jobs, int min_K,
                        int max_K, const R* d_weights, double* d_rowsum, const double* d_mode_w,
                        uint64_t* d_tab, uint64_t* d_mode_tab, int32_t* d_err, cudaStream_t s,
                        int groups_req) {
  const int cap = max_K < 64 ? 64 : max_K;
  const size_t per_group = alias_group_bytes<NW>(cap, (int)sizeof(R));
  int groups = NW == 1 ? 8 : 1;
  while (groups > 1 && per_group * groups > 96 * 1024) --groups;
  if (NW == 1 && groups_req > 0) {
    int most = 16;
    while (most > 1 && per_group * most > 200 * 1024) --most;
    groups = groups_req < most ? groups_req : most;
  }
  const size_t smem = per_group * groups;
  if (smem > 220 * 1024) return cudaErrorInvalidValue;   // rows beyond the shared-memory path
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  uint32_t blocks = (total_jobs + groups - 1) / groups;
  const uint32_t cap_blocks = (uint32_t)sms * 32;
  if (blocks > cap_blocks) blocks = cap_blocks;
  // sum-rule tolerance: FP64 weights agree with A to rounding; FP32 propagation to ~1e-5
  const double tol = sizeof(R) == 8 ? 1e-8 : 1e-3;
  const cudaError_t e = allow_smem(alias_kernel<R, NW>);
  if (e != cudaSuccess) return e;
  alias_kernel<R, NW><<<blocks, groups * 32 * NW, smem, s>>>(
      d_tasks, n_tasks, total_jobs, min_K, max_K, cap, tol, d_weights, d_rowsum, d_mode_w, d_tab,
      d_mode_tab, d_err);
  return cudaGetLastError();
}

template <typename R>
cudaError_t alias_classes(const TaskDesc* d_tasks, int n_tasks, uint32_t total_jobs, int min_K,
                          int max_K, const R* d_weights, double* d_rowsum, const double* d_mode_w,
                          uint64_t* d_tab, uint64_t* d_mode_tab, int32_t* d_err, cudaStream_t s,
                          int warps_req) {
  cudaError_t e = cudaSuccess;
  const int ends[3] = {0, kAliasShortRow, kAliasWarpRow};
  for (int c = 0; c < 2 && e == cudaSuccess; ++c)
    if (max_K > ends[c] && min_K <= ends[c + 1])
      e = alias_class<R, 1>(d_tasks, n_tasks, total_jobs, ends[c],
                            max_K < ends[c + 1] ? max_K : ends[c + 1], d_weights, d_rowsum,
                            d_mode_w, d_tab, d_mode_tab, d_err, s, warps_req);
  if (e == cudaSuccess && max_K > kAliasWarpRow)
    e = alias_class<R, 4>(d_tasks, n_tasks, total_jobs, kAliasWarpRow, max_K, d_weights, d_rowsum,
                          d_mode_w, d_tab, d_mode_tab, d_err, s, 0);
  return e;
}
}  // namespace

cudaError_t launch_alias_build(const TaskDesc* d_tasks, int n_tasks, uint32_t total_jobs,
                               int min_K, int max_K, int precision, const void* d_weights,
                               double* d_rowsum, const double* d_mode_w, uint64_t* d_tab,
                               uint64_t* d_mode_tab, int32_t* d_err, cudaStream_t s,
                               int warps_req) {
  if (total_jobs == 0) return cudaSuccess;
  if (precision == NEGF_FP64)
    return alias_classes<double>(d_tasks, n_tasks, total_jobs, min_K, max_K,
                                 static_cast<const double*>(d_weights), d_rowsum, d_mode_w, d_tab,
                                 d_mode_tab, d_err, s, warps_req);
  return alias_classes<float>(d_tasks, n_tasks, total_jobs, min_K, max_K,
                              static_cast<const float*>(d_weights), d_rowsum, d_mode_w, d_tab,
                              d_mode_tab, d_err, s, warps_req);
}

}  // namespace negf
