// Linear conductance with continuous energies: each walker draws its energy from the thermal
// window Th(E) = -df/dE (Eq. Gqp_expression; the sampling density of Eq. gpq_formula) restricted
// to the span of a wire's energy grid, and walks the Step 6' chain whose transition
// probabilities are interpolated linearly between the two grid energies around it (the
// interpolation of the p_i in the paper's Sec. "Interpolation"): each draw takes the upper grid
// energy's alias table with probability alpha, else the lower one's (an interval where the start
// lead has no open channel at one end walks with the other end's table).  A walker absorbed at
// q = 1 - p scores c(E) = (1 - alpha) c_i + alpha c_{i+1} (Eq. elast_lin_xpq); the tally keeps,
// per grid interval, the absorbed count, sum of a = floor(alpha 2^32) and sum of (a >> 16)^2 in
// integers, from which the host forms the mean and variance of the score exactly.
//
// Random numbers (Philox4x32-10, counter (b, id_lo, id_hi, 0x80000000 | wire)): block 0 -> the
// energy (x0, x1: a 53-bit word v whose CDF value F = F0 + (v + 1/2) 2^-53 window gives the
// interval, found by comparing v with the host's integer thresholds of the grid points, and
// the energy) and the injection table (x2); block 1 -> the injection mode (x0, x1); block
// b >= 2 -> transition b - 1, (x0, x1) on the row (two-level tables: on the level-1 row, and x3
// for the site within a drawn slice) and x2 < a for the table.
//
// What bounds it: the setup of a walker (two Philox blocks, the interval search, FP64 steps on a
// narrow pipe, two logarithms) costs about as much as two transitions, and walks differ in
// length.  A warp works through chunks of consecutive walkers; once half of its lanes are idle
// they are set up together, so that neither the setup runs for a few lanes nor a warp waits for
// its longest walk.  What depends on the grid interval alone (its energies relative to mu,
// thresholds, open ends, table offsets) is staged in shared memory once per block.  The block's
// tally sits in shared memory too and is added to global memory once.  W=10 x L=50, 132 energies,
// 1.6e7 walkers: 1.21 -> 0.76 ms against a walker per thread and stride of the grid.
//
// Staging takes 88 bytes of shared memory an interval (the tally alone 24) and time per block, and
// the votes of a warp lengthen every step of a lone walk.  Launches of few walkers and grids that
// would leave fewer than four blocks an SM take thermal_few_kernel instead (which, and both
// sides' times: launch_thermal_walk).
#include <cuda_runtime.h>
#include <math.h>

#include "negf_internal.cuh"
#include "philox.cuh"

namespace negf {
namespace {

constexpr int kThermalThreads = 256;

// A grid interval: the threshold of its upper end, its table offsets (one-level rows, or level-1
// rows, and the level-2 blocks), E_i - mu and E_{i+1} - E_i, mode rows, whether the start lead
// has an open channel at either end.
struct ThermalInterval {
  unsigned long long thr;
  uint64_t tab_lo, tab_hi, l2_lo, l2_hi;
  float e0, de;
  uint32_t mode_lo, mode_hi;
  bool open_lo, open_hi;
};

// Interval e of the grid of tasks task0 ..; thr and open channels of lead p
__device__ __forceinline__ ThermalInterval thermal_interval(const TaskDesc* __restrict__ tasks,
                                                            int task0, int e, bool two,
                                                            const double* __restrict__ cvals, int p,
                                                            double mu, unsigned long long thr) {
  const TaskDesc &da = tasks[task0 + e], &db = tasks[task0 + e + 1];
  ThermalInterval iv;
  iv.thr = thr;
  iv.tab_lo = two ? da.l1_off : da.tab_off;
  iv.tab_hi = two ? db.l1_off : db.tab_off;
  iv.l2_lo = da.tab_off;
  iv.l2_hi = db.tab_off;
  iv.e0 = (float)(da.E - mu);
  iv.de = (float)(db.E - da.E);
  iv.mode_lo = da.mode_off;
  iv.mode_hi = db.mode_off;
  iv.open_lo = cvals[2 * (task0 + e) + p] > 0.0;
  iv.open_hi = cvals[2 * (task0 + e + 1) + p] > 0.0;
  return iv;
}

// The word a = floor(alpha 2^32) of the energy of CDF value pE in interval `in`:
// E - E_i = kT ln(F / (1 - F)) - (E_i - mu), the logarithms in FP32 of F and 1 - F (the latter
// formed in FP64, so that both keep their relative precision); alpha to ~2^-20
__device__ __forceinline__ uint32_t thermal_alpha(double pE, double kT, const ThermalInterval& in) {
  const float lnr = logf((float)pE) - logf((float)(1.0 - pE));
  const float dE = (float)kT * lnr - in.e0;
  float alpha = dE / in.de;
  alpha = alpha < 0.f ? 0.f : (alpha > 1.f ? 1.f : alpha);
  const float af = floorf(alpha * 4294967296.f);
  return af >= 4294967295.f ? 0xffffffffu : (uint32_t)af;
}

// The site drawn within slice k of a row's level-2 blocks (v = 31 random bits): the index of the
// next row
__device__ __forceinline__ uint32_t thermal_site(const uint64_t* __restrict__ blocks, uint32_t row,
                                                 uint32_t k, uint32_t L, uint32_t W, uint32_t B2,
                                                 uint32_t v) {
  const uint4* blk =
      reinterpret_cast<const uint4*>(blocks) + (((uint64_t)row * L + k) * B2 >> 2);
  uint32_t oct = 0;
  if (W > 8) {
    const uint4 q0 = __ldg(blk), q1 = __ldg(blk + 1);
    oct = (q0.x <= v) + (q0.y <= v) + (q0.z <= v) + (q0.w <= v) + (q1.x <= v) + (q1.y <= v) +
          (q1.z <= v) + (q1.w <= v);
    blk += 2 + 2 * oct;
  }
  const uint4 o0 = __ldg(blk), o1 = __ldg(blk + 1);
  return k * W + 8 * oct + (o0.x <= v) + (o0.y <= v) + (o0.z <= v) + (o0.w <= v) + (o1.x <= v) +
         (o1.y <= v) + (o1.z <= v) + (o1.w <= v);
}

__device__ __forceinline__ void smem_add64(unsigned* lohi, unsigned v) {
  const unsigned old = atomicAdd(lohi, v);
  if (old + v < old) atomicAdd(lohi + 1, 1u);
}
// 64-bit add to a shared counter kept as two 32-bit words
__device__ __forceinline__ void add64(unsigned* lohi, uint64_t v) {
  if (v == 0) return;
  smem_add64(lohi, (unsigned)v);
  if (v >> 32) atomicAdd(lohi + 1, (unsigned)(v >> 32));
}

// Per-interval sums of the walks just absorbed at q, lanes `done` (the calling lane among them):
// lanes with the same interval pool theirs and one of them adds them
__device__ __forceinline__ void thermal_add(unsigned* s_t, unsigned done, int iv, uint32_t a) {
  const unsigned grp = __match_any_sync(done, iv);
  const uint32_t a16 = a >> 16, sq = a16 * a16;
  const uint32_t cnt = __popc(grp);
  const uint32_t a_hi = __reduce_add_sync(grp, a >> 16), a_lo = __reduce_add_sync(grp, a & 0xffffu);
  const uint32_t s_hi = __reduce_add_sync(grp, sq >> 16), s_lo = __reduce_add_sync(grp, sq & 0xffffu);
  if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
    smem_add64(&s_t[2 * (3 * iv + 0)], cnt);
    add64(&s_t[2 * (3 * iv + 1)], ((uint64_t)a_hi << 16) + a_lo);
    add64(&s_t[2 * (3 * iv + 2)], ((uint64_t)s_hi << 16) + s_lo);
  }
}

// kTwo: the grid's tables are two-level (level 1 an alias row over the slices and leads, level 2
// the inverse-CDF blocks of the slices): a transition draws the slice or lead with (x0, x1),
// the table with x2, and the site within the slice with x3 (v = x3 >> 1).
template <bool kTwo>
__global__ void __launch_bounds__(kThermalThreads) thermal_walk_kernel(
    const TaskDesc* __restrict__ tasks, int task0, int M, uint32_t wire,
    const uint64_t* __restrict__ tab, const uint64_t* __restrict__ mode_tab,
    const double* __restrict__ cvals, int p, PhiloxKey key, uint64_t walkers, uint64_t id_offset,
    uint32_t max_steps, double mu, double kT, double F0, double window,
    const unsigned long long* __restrict__ thr, unsigned long long* __restrict__ tally,
    int32_t* __restrict__ t_lead,
    uint32_t* __restrict__ t_steps, int32_t* __restrict__ t_interval, uint32_t* __restrict__ t_a,
    unsigned chunk_size) {
  // shared tally: per interval (absorbed at q, sum a, sum (a >> 16)^2), then absorbed L, R,
  // closed, truncated, steps; each a 64-bit counter kept as two 32-bit words; before it the
  // intervals' data
  extern __shared__ __align__(16) unsigned char s_raw[];
  ThermalInterval* s_iv = reinterpret_cast<ThermalInterval*>(s_raw);       // [M - 1]
  unsigned* s_t = reinterpret_cast<unsigned*>(s_iv + (M - 1));
  const int n_fields = 3 * (M - 1) + 5;
  for (int i = threadIdx.x; i < 2 * n_fields; i += blockDim.x) s_t[i] = 0u;
  for (int e = threadIdx.x; e < M - 1; e += blockDim.x)
    s_iv[e] = thermal_interval(tasks, task0, e, kTwo, cvals, p, mu, thr[e]);
  __syncthreads();
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int q = 1 - p;
  const int G0 = 3 * (M - 1);
  const uint32_t ctr3 = 0x80000000u | wire;
  const TaskDesc& d0 = tasks[task0];
  const uint32_t n = (uint32_t)d0.n, W = (uint32_t)d0.W, K = (uint32_t)d0.K;
  const uint32_t L = (uint32_t)d0.L, K1 = kTwo ? L + 2 : K, B2 = (uint32_t)level2_words(d0.W);
  uint64_t my_abs0 = 0, my_abs1 = 0, my_closed = 0, my_trunc = 0, my_steps = 0;
  // chunks of consecutive walkers, strided over the grid's warps
  const uint64_t stride = (uint64_t)gridDim.x * (kThermalThreads / 32) * chunk_size;
  uint64_t chunk = ((uint64_t)blockIdx.x * (kThermalThreads / 32) + (threadIdx.x >> 5)) * chunk_size;
  unsigned taken = 0;                                 // walkers of the chunk handed out
  // the walk in flight
  bool has = false, mix = false, open_hi = false;
  uint64_t g = 0;
  uint32_t lo = 0, hi = 0, a = 0, b = 0, row = 0, steps = 0;
  int iv = 0;
  auto upper = [&](uint32_t word) { return mix ? word < a : open_hi; };
  auto finish = [&](int outcome) {
    if (outcome == 0) ++my_abs0;
    else if (outcome == 1) ++my_abs1;
    else if (outcome == -1) ++my_closed;
    else ++my_trunc;
    my_steps += steps;
    if (t_lead) t_lead[g] = outcome;
    if (t_steps) t_steps[g] = steps;
    if (t_interval) t_interval[g] = iv;
    if (t_a) t_a[g] = a;
    has = false;
  };
  while (true) {
    // ---- set up new walkers once half of the lanes are idle (or nothing else is left)
    const unsigned idle = __ballot_sync(FULL, !has);
    if (chunk < walkers && (__popc(idle) >= 16 || idle == FULL)) {
      const unsigned size =
          walkers - chunk < chunk_size ? (unsigned)(walkers - chunk) : chunk_size;
      const unsigned mine = taken + __popc(idle & lt_mask);
      taken += __popc(idle);
      if (!has && mine < size) {
        g = chunk + mine;
        const uint64_t wid = id_offset + g;
        lo = (uint32_t)wid;
        hi = (uint32_t)(wid >> 32);
        const uint4 r0 = philox4x32_10(make_uint4(0u, lo, hi, ctr3), key);
        const uint64_t v = (((uint64_t)r0.x << 32) | r0.y) >> 11;
        const double u = ((double)v + 0.5) * 0x1p-53;
        const double pE = F0 + u * window;                // F(E) of the drawn energy
        // last grid index with F(E_e) <= F(E): the number of grid points 1 .. M - 1 whose
        // threshold v reaches (an integer search, no FP64 compares)
        int lo_i = 0, hi_i = M - 1;
        while (lo_i < hi_i) {
          const int mid = (lo_i + hi_i) >> 1;
          if (s_iv[mid].thr <= v) lo_i = mid + 1; else hi_i = mid;
        }
        iv = lo_i < M - 2 ? lo_i : M - 2;
        const ThermalInterval& in = s_iv[iv];
        a = thermal_alpha(pE, kT, in);
        // an interval open at both ends mixes the two tables; one open at a single end walks
        // with that end's table alone (a chain without an open lead never absorbs)
        open_hi = in.open_hi;
        mix = in.open_lo && in.open_hi;
        steps = 0;
        if (in.open_lo || in.open_hi) {
          const uint4 r1 = philox4x32_10(make_uint4(1u, lo, hi, ctr3), key);
          const uint64_t* mrow = mode_tab + (upper(r0.z) ? in.mode_hi : in.mode_lo) + p * W;
          const uint32_t c = __umulhi(r1.x, W);
          const uint64_t e = __ldg(mrow + c);
          row = n + p * W + (r1.y < (uint32_t)e ? c : (uint32_t)(e >> 32));
          b = 2;
          has = true;
        } else {
          finish(-1);
        }
      }
      if (taken >= size) {
        chunk += stride;
        taken = 0;
      }
    } else if (idle == FULL) {
      break;
    }
    // ---- one transition of every walk in flight
    bool absorbed = false;                               // at q
    if (has) {
      const ThermalInterval& in = s_iv[iv];
      const uint4 r = philox4x32_10(make_uint4(b, lo, hi, ctr3), key);
      ++b;
      const bool up = upper(r.z);
      const uint32_t cc = __umulhi(r.x, K1);
      const uint64_t ee = __ldg(tab + (up ? in.tab_hi : in.tab_lo) + (uint64_t)row * K1 + cc);
      uint32_t j = r.y < (uint32_t)ee ? cc : (uint32_t)(ee >> 32);
      if (kTwo) {
        const uint32_t k = j;
        if (k >= L) {
          j = n + (k - L);
        } else {
          j = thermal_site(tab + (up ? in.l2_hi : in.l2_lo), row, k, L, W, B2, r.w >> 1);
        }
      }
      ++steps;
      if (j >= n) {
        absorbed = (int)(j - n) == q;
        finish((int)(j - n));
      } else if (steps >= max_steps) {
        finish(-2);
      } else {
        row = j;
      }
    }
    const unsigned done = __ballot_sync(FULL, absorbed);
    if (absorbed) thermal_add(s_t, done, iv, a);
  }
  add64(&s_t[2 * (G0 + 0)], my_abs0);
  add64(&s_t[2 * (G0 + 1)], my_abs1);
  add64(&s_t[2 * (G0 + 2)], my_closed);
  add64(&s_t[2 * (G0 + 3)], my_trunc);
  add64(&s_t[2 * (G0 + 4)], my_steps);
  __syncthreads();
  for (int f = threadIdx.x; f < n_fields; f += blockDim.x) {
    const unsigned long long v = ((unsigned long long)s_t[2 * f + 1] << 32) | s_t[2 * f];
    if (v) atomicAdd(tally + f, v);
  }
}

// The same walks where walkers are few or the grid is large: the intervals' data is read where a
// walker is set up (only the tally takes shared memory), and once nothing is left to hand out
// every lane goes on alone, without the warp's votes, the next Philox block drawn while a
// table entry is fetched.  Four blocks an SM: with five, 48 registers, a lone walk's step
// takes 30 % longer.
template <bool kTwo>
__global__ void __launch_bounds__(kThermalThreads, 4) thermal_few_kernel(
    const TaskDesc* __restrict__ tasks, int task0, int M, uint32_t wire,
    const uint64_t* __restrict__ tab, const uint64_t* __restrict__ mode_tab,
    const double* __restrict__ cvals, int p, PhiloxKey key, uint64_t walkers, uint64_t id_offset,
    uint32_t max_steps, double mu, double kT, double F0, double window,
    const unsigned long long* __restrict__ thr, unsigned long long* __restrict__ tally,
    int32_t* __restrict__ t_lead,
    uint32_t* __restrict__ t_steps, int32_t* __restrict__ t_interval, uint32_t* __restrict__ t_a,
    unsigned chunk_size) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  unsigned* s_t = reinterpret_cast<unsigned*>(s_raw);                      // the tally, as above
  const int n_fields = 3 * (M - 1) + 5;
  for (int i = threadIdx.x; i < 2 * n_fields; i += blockDim.x) s_t[i] = 0u;
  __syncthreads();
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int q = 1 - p;
  const int G0 = 3 * (M - 1);
  const uint32_t ctr3 = 0x80000000u | wire;
  const TaskDesc& d0 = tasks[task0];
  const uint32_t n = (uint32_t)d0.n, W = (uint32_t)d0.W, K = (uint32_t)d0.K;
  const uint32_t L = (uint32_t)d0.L, K1 = kTwo ? L + 2 : K, B2 = (uint32_t)level2_words(d0.W);
  uint64_t my_abs0 = 0, my_abs1 = 0, my_closed = 0, my_trunc = 0, my_steps = 0;
  const uint64_t stride = (uint64_t)gridDim.x * (kThermalThreads / 32) * chunk_size;
  uint64_t chunk = ((uint64_t)blockIdx.x * (kThermalThreads / 32) + (threadIdx.x >> 5)) * chunk_size;
  unsigned taken = 0;                                 // walkers of the chunk handed out
  // the walk in flight, its tables and (ended at q, not in the tally yet) whether it was absorbed
  bool has = false, mix = false, open_hi = false, absorbed = false;
  uint64_t g = 0;
  uint32_t lo = 0, hi = 0, a = 0, b = 0, row = 0, steps = 0;
  const uint64_t *t_lo = tab, *t_hi = tab, *l2_lo = tab, *l2_hi = tab;
  int iv = 0;
  auto upper = [&](uint32_t word) { return mix ? word < a : open_hi; };
  auto draw = [&](uint32_t at) { return philox4x32_10(make_uint4(at, lo, hi, ctr3), key); };
  auto finish = [&](int outcome) {
    if (outcome == 0) ++my_abs0;
    else if (outcome == 1) ++my_abs1;
    else if (outcome == -1) ++my_closed;
    else ++my_trunc;
    my_steps += steps;
    if (t_lead) t_lead[g] = outcome;
    if (t_steps) t_steps[g] = steps;
    if (t_interval) t_interval[g] = iv;
    if (t_a) t_a[g] = a;
    has = false;
    absorbed = outcome == q;
  };
  // one transition from Philox block r; meanwhile() runs while the table entry is fetched
  auto step = [&](const uint4 r, auto meanwhile) {
    const bool up = upper(r.z);
    const uint32_t cc = __umulhi(r.x, K1);
    const uint64_t ee = __ldg((up ? t_hi : t_lo) + (uint64_t)row * K1 + cc);
    meanwhile();
    uint32_t j = r.y < (uint32_t)ee ? cc : (uint32_t)(ee >> 32);
    if (kTwo) {
      const uint32_t k = j;
      j = k >= L ? n + (k - L)
                 : thermal_site(up ? l2_hi : l2_lo, row, k, L, W, B2, r.w >> 1);
    }
    ++steps;
    if (j >= n) finish((int)(j - n));
    else if (steps >= max_steps) finish(-2);
    else row = j;
  };
  while (chunk < walkers) {
    // ---- set up new walkers once 20 lanes are idle
    const unsigned idle = __ballot_sync(FULL, !has);
    if (__popc(idle) >= 20) {
      const unsigned size =
          walkers - chunk < chunk_size ? (unsigned)(walkers - chunk) : chunk_size;
      const unsigned mine = taken + __popc(idle & lt_mask);
      taken += __popc(idle);
      if (!has && mine < size) {
        g = chunk + mine;
        const uint64_t wid = id_offset + g;
        lo = (uint32_t)wid;
        hi = (uint32_t)(wid >> 32);
        const uint4 r0 = draw(0u);
        const uint64_t v = (((uint64_t)r0.x << 32) | r0.y) >> 11;
        const double u = ((double)v + 0.5) * 0x1p-53;
        const double pE = F0 + u * window;                // F(E) of the drawn energy
        int lo_i = 0, hi_i = M - 1;                       // the interval, as above
        while (lo_i < hi_i) {
          const int mid = (lo_i + hi_i) >> 1;
          if (thr[mid] <= v) lo_i = mid + 1; else hi_i = mid;
        }
        iv = lo_i < M - 2 ? lo_i : M - 2;
        const ThermalInterval in = thermal_interval(tasks, task0, iv, kTwo, cvals, p, mu, 0ull);
        a = thermal_alpha(pE, kT, in);
        open_hi = in.open_hi;
        mix = in.open_lo && in.open_hi;
        t_lo = tab + in.tab_lo;
        t_hi = tab + in.tab_hi;
        l2_lo = tab + in.l2_lo;
        l2_hi = tab + in.l2_hi;
        steps = 0;
        if (in.open_lo || in.open_hi) {
          const uint4 r1 = draw(1u);
          const uint64_t* mrow = mode_tab + (upper(r0.z) ? in.mode_hi : in.mode_lo) + p * W;
          const uint32_t c = __umulhi(r1.x, W);
          const uint64_t e = __ldg(mrow + c);
          row = n + p * W + (r1.y < (uint32_t)e ? c : (uint32_t)(e >> 32));
          b = 2;
          has = true;
        } else {
          finish(-1);
        }
      }
      if (taken >= size) {
        chunk += stride;
        taken = 0;
      }
      if (chunk >= walkers) break;
    }
    // ---- one transition of every walk in flight
    if (has) {
      const uint4 r = draw(b++);
      step(r, [] {});
    }
    const unsigned done = __ballot_sync(FULL, absorbed);
    if (absorbed) thermal_add(s_t, done, iv, a);
    absorbed = false;
  }
  // ---- nothing left to hand out: every walk to its end
  if (has) {
    uint4 r = draw(b);
    while (has) {
      uint4 next;
      step(r, [&] { next = draw(++b); });
      r = next;
    }
  }
  __syncwarp();
  const unsigned done = __ballot_sync(FULL, absorbed);
  if (absorbed) thermal_add(s_t, done, iv, a);
  add64(&s_t[2 * (G0 + 0)], my_abs0);
  add64(&s_t[2 * (G0 + 1)], my_abs1);
  add64(&s_t[2 * (G0 + 2)], my_closed);
  add64(&s_t[2 * (G0 + 3)], my_trunc);
  add64(&s_t[2 * (G0 + 4)], my_steps);
  __syncthreads();
  for (int f = threadIdx.x; f < n_fields; f += blockDim.x) {
    const unsigned long long v = ((unsigned long long)s_t[2 * f + 1] << 32) | s_t[2 * f];
    if (v) atomicAdd(tally + f, v);
  }
}

}  // namespace

// ---- interval distances of the interpolating sampler's grid (Sec. "Interpolation") ----------
// For consecutive grid energies e, e + 1 of one wire: d_e = the largest of the rows' total-
// variation distances (1/2) sum_b |w_ab(e) / S_a(e) - w_ab(e+1) / S_a(e+1)| (S the FP64 row
// sums; a row of zero sum counts as all zeros), the same between the injection-mode
// distributions of lead p, and |c_e - c_{e+1}| / max(c_e, c_{e+1}).  One warp per (interval,
// row), FP64 sums; d (doubles >= 0, zeroed by the caller) takes the maximum through atomicMax
// on the bit patterns, which order like the values for non-negative doubles.
namespace {
template <typename R>
__global__ void interval_distance_kernel(const TaskDesc* __restrict__ tasks, int task0, int M,
                                         const R* __restrict__ weights,
                                         const double* __restrict__ rowsum,
                                         const double* __restrict__ mode_w,
                                         const double* __restrict__ cvals, int p,
                                         unsigned long long* __restrict__ d) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const TaskDesc& t0 = tasks[task0];
  const int rows = t0.rows, K = t0.K, W = t0.W;
  const int per = rows + 1;                           // the rows, then the modes and c
  if (warp >= (M - 1) * per) return;
  const int e = warp / per, row = warp - e * per;
  const TaskDesc& da = tasks[task0 + e];
  const TaskDesc& db = tasks[task0 + e + 1];
  double tv = 0.0;
  if (row < rows) {
    const double sa = rowsum[da.row_base + row], sb = rowsum[db.row_base + row];
    const double ia = sa > 0.0 ? 1.0 / sa : 0.0, ib = sb > 0.0 ? 1.0 / sb : 0.0;
    const R* wa = weights + da.wt_off + (uint64_t)row * K;
    const R* wb = weights + db.wt_off + (uint64_t)row * K;
    for (int j = lane; j < K; j += 32) tv += fabs((double)wa[j] * ia - (double)wb[j] * ib);
  } else {
    const double* ma = mode_w + da.mode_off + p * W;
    const double* mb = mode_w + db.mode_off + p * W;
    double sa = 0.0, sb = 0.0;
    for (int j = 0; j < W; ++j) {
      sa += ma[j];
      sb += mb[j];
    }
    const double ia = sa > 0.0 ? 1.0 / sa : 0.0, ib = sb > 0.0 ? 1.0 / sb : 0.0;
    for (int j = lane; j < W; j += 32) tv += fabs(ma[j] * ia - mb[j] * ib);
  }
  for (int o = 16; o > 0; o >>= 1) tv += __shfl_down_sync(0xffffffffu, tv, o);
  if (lane == 0) {
    double v = 0.5 * tv;
    if (row == rows) {
      const double ca = cvals[2 * (task0 + e) + p], cb = cvals[2 * (task0 + e + 1) + p];
      const double cm = fmax(ca, cb);
      if (cm > 0.0) v = fmax(v, fabs(ca - cb) / cm);
    }
    atomicMax(d + e, (unsigned long long)__double_as_longlong(v));
  }
}

}  // namespace

cudaError_t launch_interval_distance(const TaskDesc* d_tasks, int task0, int M, int rows,
                                     int precision, const void* d_weights,
                                     const double* d_rowsum, const double* d_mode_w,
                                     const double* d_c, int start_lead, double* d_out,
                                     cudaStream_t s) {
  if (M < 2) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(d_out, 0, sizeof(double) * (M - 1), s);
  if (e != cudaSuccess) return e;
  const uint64_t warps = (uint64_t)(M - 1) * (rows + 1);
  const unsigned blocks = (unsigned)((warps + 7) / 8);
  auto* o = reinterpret_cast<unsigned long long*>(d_out);
  if (precision == NEGF_FP64)
    interval_distance_kernel<double><<<blocks, 256, 0, s>>>(
        d_tasks, task0, M, static_cast<const double*>(d_weights), d_rowsum, d_mode_w, d_c,
        start_lead, o);
  else
    interval_distance_kernel<float><<<blocks, 256, 0, s>>>(
        d_tasks, task0, M, static_cast<const float*>(d_weights), d_rowsum, d_mode_w, d_c,
        start_lead, o);
  return cudaGetLastError();
}

cudaError_t launch_thermal_walk(const TaskDesc* d_tasks, int task0, int M, int wire,
                                const uint64_t* d_tab, const uint64_t* d_mode_tab,
                                const double* d_c, int start_lead, uint64_t seed,
                                uint64_t walkers, uint64_t id_offset, uint32_t max_steps,
                                double mu, double kT, double F0, double window,
                                const unsigned long long* d_thr, unsigned long long* d_tally,
                                int32_t* d_lead, uint32_t* d_steps, int32_t* d_interval,
                                uint32_t* d_a, int sm_count, cudaStream_t s, bool two_level) {
  if (walkers == 0 || M < 2) return cudaSuccess;
  const PhiloxKey key{(uint32_t)seed, (uint32_t)(seed >> 32)};
  // Which kernel (GB300, us of the kernel; "before" a walker per thread and stride of the grid):
  // * grids of more than 651 intervals: staged, fewer than four blocks fit an SM.  W=4 x L=10,
  //   1.6e7 walkers: 1000 energies 914 staged, 683 few (before 657), 2046 energies 1728, 856 (780);
  //   W=10 x L=50, 1000 energies 1306, 949 (1452);
  // * up to three walkers a lane (four blocks an SM; 466,944 walkers on 152 SMs): a lone walk's
  //   latency counts.  W=3 x L=150, 9 energies, 1e5 walkers 195, 109 (before 134), 5e5 267, 170
  //   (226); W=4 x L=10 1e5 17, 16 (17), 5e5 33, 38 (31).
  // The staging kernel takes the blocks that fit while a lane has fewer than eight walkers (those
  // of a second round would wait for the first: W=10 x L=50, 9 energies, 7e5 walkers 73 -> 65), and
  // more beyond, which evens out the ends of the blocks (4e6 walkers 201 -> 188).  The few kernel
  // takes the blocks that fit, or up to half as many more if each lane then has one walker.
  const size_t tally = sizeof(unsigned) * 2 * (size_t)(3 * (M - 1) + 5);
  const size_t staged = tally + sizeof(ThermalInterval) * (size_t)(M - 1);
  constexpr size_t kStagedMost = 56 * 1024;
  const uint64_t lanes = (uint64_t)sm_count * 4 * kThermalThreads;
  const bool few = staged > kStagedMost || walkers <= 3 * lanes;
  const size_t smem = few ? tally : staged;
  auto kern = two_level ? (few ? thermal_few_kernel<true> : thermal_walk_kernel<true>)
                        : (few ? thermal_few_kernel<false> : thermal_walk_kernel<false>);
  cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  int per_sm = 8;
  if (few || walkers < 8 * lanes) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThermalThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
  }
  const uint64_t need = (walkers + kThermalThreads - 1) / kThermalThreads;
  uint64_t blocks = (uint64_t)sm_count * per_sm;
  if (blocks > need || (few && 2 * need <= 3 * blocks)) blocks = need;
  const uint64_t warps = blocks * (kThermalThreads / 32);
  unsigned chunk = walk_chunk(walkers, warps);
  if (few && chunk == 512) {
    // equal chunks: with as many blocks as fit, a share of 513 walkers in chunks of 512 would give
    // some warps twice the walks of the others (4e6 walkers, 1000 energies: 207 -> 193)
    const uint64_t per = (walkers + warps - 1) / warps, n = (per + 511) / 512;
    chunk = (unsigned)(((per + n - 1) / n + 31) / 32 * 32);
  }
  kern<<<(unsigned)blocks, kThermalThreads, smem, s>>>(
      d_tasks, task0, M, (uint32_t)wire, d_tab, d_mode_tab, d_c, start_lead, key, walkers,
      id_offset, max_steps, mu, kT, F0, window, d_thr, d_tally, d_lead, d_steps, d_interval,
      d_a, chunk);
  return cudaGetLastError();
}

}  // namespace negf
