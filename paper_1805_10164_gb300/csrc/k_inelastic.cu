// Walks with inelastic Buttiker probes: Step 6' followed by the energy draw of Step 7'
// (Sec. II.F, Eq. draw_E_last).
//
// A walker is injected from lead p at the energy of its task (Step 4, the task's mode alias
// row) and carries its current energy e with its table row.  Philox4x32-10 block b of walker
// wid has counter (b, wid_lo, wid_hi, task) and key (seed_lo, seed_hi), task the injection
// task's number: block 0 is the injection draw (words x0, x1 over the W modes); block s >= 1 is
// transition s: words (x0, x1) draw the next index from the row at energy e (alias over the
// K = n + 2 columns, leads n and n + 1), and when that is a site j, words (x2, x3) draw the
// next energy e' from the energy row (j, e) built by energy_alias_kernel
// (w_e' K(E_e' - E_e) A_jj(E_e'), the model's lambda~ of Eq. condition4_buttiker).  A draw with
// words (x, y) over a K-entry row takes c = (x K) >> 32 and keeps c if y < thr[c], else
// alias[c].  Drawing a lead ends the walk; its count goes to the injection task, so that
// T_qp(E_0) = c_p(E_0) P(q | p, E_0) as for elastic walks.  Warps take chunks of consecutive
// walkers and refill their lanes from them (below); counts per task in a lane's registers, then
// in shared memory (tasks of the launch window), added to the global tally once per block.
#include <cuda_runtime.h>

#include "negf_internal.cuh"
#include "philox.cuh"

namespace negf {
namespace {

constexpr int kThreads = 256;
constexpr int kFields = NEGF_TALLY_FIELDS;   // done, absorbed L, absorbed R, truncated, steps
constexpr int kWindow = 1024;                // injection tasks per launch (40 KB shared tally)

constexpr unsigned kFlushAt = 1u << 26;      // flush a lane's counters before they can overflow

// 64-bit counters in shared memory as (lo, hi) words: each addition carries its own overflow
__device__ __forceinline__ void add64(unsigned* lohi, unsigned v) {
  const unsigned old = atomicAdd(lohi, v);
  if (old + v < old) atomicAdd(lohi + 1, 1u);
}

// A warp works through chunks of consecutive walkers (chunk numbers strided over the grid's
// warps, so that the walks in flight share a few tasks' tables); a lane whose walk has ended
// takes the chunk's next walker, so that a warp does not wait for its longest walk.  Every
// iteration spends one Philox block per walk: the injection draw, or a transition with its
// energy draw.  Counts stay in registers while a lane's walkers belong to one task: added to
// the block's shared tally per walk, three same-address shared atomics a walk serialised over
// the warp's lanes and bounded the kernel (W=10 x L=50, 64 energies, 1e6 walkers each:
// 3.64 -> 1.62 ms; what is left is the latency of the two dependent gathers).
__global__ void __launch_bounds__(kThreads) inelastic_walk_kernel(
    const TaskDesc* __restrict__ tasks, int task0, int n_tasks,
    const EnergyDesc* __restrict__ edesc, const uint64_t* __restrict__ tab,
    const uint64_t* __restrict__ mode_tab, const double* __restrict__ cvals,
    const uint64_t* __restrict__ etab, int start_lead, PhiloxKey key, uint64_t walkers_per_task,
    uint64_t id_offset, uint32_t max_steps, unsigned long long* __restrict__ tally,
    unsigned chunk_size) {
  extern __shared__ unsigned s_tally[];                        // [task][field][lo, hi]
  for (int i = threadIdx.x; i < n_tasks * kFields * 2; i += blockDim.x) s_tally[i] = 0u;
  __syncthreads();
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const unsigned long long total = (unsigned long long)n_tasks * walkers_per_task;
  const unsigned long long stride =
      (unsigned long long)gridDim.x * (kThreads / 32) * chunk_size;
  unsigned long long chunk =
      ((unsigned long long)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * chunk_size;
  unsigned taken = 0;                        // walkers of the chunk handed out
  // the lane's task (counts a not yet in shared memory) and what its walks need of it
  int tl = -1;
  unsigned long long t_first = 0;
  unsigned a[kFields] = {0u, 0u, 0u, 0u, 0u};
  bool open = false;
  uint32_t task_id = 0, n = 0, K = 0, W = 0, nE = 0;
  const uint64_t* mrow = nullptr;
  // tables and energy rows of the wire's first energy and their strides from one energy to the
  // next (a wire's tasks are consecutive and alike)
  const uint64_t *trow0 = nullptr, *erow0 = nullptr;
  uint64_t t_stride = 0, e_stride = 0;
  uint32_t e0 = 0;                           // the task's own energy index
  // the walk in flight: energy index, row, Philox block, steps
  bool has = false;
  uint32_t wlo = 0, whi = 0, e = 0, row = 0, b = 0, steps = 0;
  auto flush = [&]() {
    unsigned* t = s_tally + tl * kFields * 2;
#pragma unroll
    for (int f = 0; f < kFields; ++f) {
      if (a[f]) add64(t + 2 * f, a[f]);
      a[f] = 0u;
    }
  };
  while (true) {
    const unsigned idle = __ballot_sync(FULL, !has);
    if (idle) {
      if (chunk < total) {
        const unsigned size =
            total - chunk < chunk_size ? (unsigned)(total - chunk) : chunk_size;
        const unsigned mine = taken + __popc(idle & lt_mask);
        taken += __popc(idle);
        if (!has && mine < size) {
          const unsigned long long g = chunk + mine;
          if (tl < 0 || g - t_first >= walkers_per_task) {
            if (tl >= 0) flush();
            tl = (int)(g / walkers_per_task);
            t_first = (unsigned long long)tl * walkers_per_task;
            const int t = task0 + tl;
            const TaskDesc& d = tasks[t];
            const EnergyDesc ed = edesc[t];
            task_id = (uint32_t)t;
            n = (uint32_t)d.n;
            K = (uint32_t)d.K;
            W = (uint32_t)d.W;
            nE = (uint32_t)ed.nE;
            e0 = (uint32_t)(t - ed.t0);
            mrow = mode_tab + d.mode_off + start_lead * d.W;
            trow0 = tab + tasks[ed.t0].tab_off;
            erow0 = etab + edesc[ed.t0].eoff;
            t_stride = (uint64_t)d.rows * d.K;
            e_stride = (uint64_t)d.n * ed.nE;
            open = cvals[2 * t + start_lead] > 0.0;
          }
          if (open) {
            const uint64_t w = id_offset + (g - t_first);
            wlo = (uint32_t)w;
            whi = (uint32_t)(w >> 32);
            e = e0;
            b = steps = 0u;
            has = true;
          } else {
            a[0] += 1u;                      // no open channel: nothing to inject
          }
        }
        if (taken >= size) {
          chunk += stride;
          taken = 0;
        }
      } else if (idle == FULL) {
        break;
      }
    }
    if (!has) continue;
    const uint4 r = philox4x32_10(make_uint4(b, wlo, whi, task_id), key);
    // block 0: the injection mode at the task's energy; block s: transition s
    const bool inject = b == 0u;
    const uint32_t c = __umulhi(r.x, inject ? W : K);
    const uint64_t* src = inject ? mrow : trow0 + e * t_stride + (uint64_t)row * K;
    const uint64_t ent = __ldg(src + c);
    const uint32_t j = r.y < (uint32_t)ent ? c : (uint32_t)(ent >> 32);
    ++b;
    if (inject) {
      row = n + start_lead * W + j;
      continue;
    }
    ++steps;
    if (j < n && steps < max_steps) {
      // Step 7': the next energy from the energy row (j, e)
      const uint32_t ce = __umulhi(r.z, nE);
      const uint64_t ee = __ldg(erow0 + e * e_stride + (uint64_t)j * nE + ce);
      e = r.w < (uint32_t)ee ? ce : (uint32_t)(ee >> 32);
      row = j;
      continue;
    }
    has = false;
    a[0] += 1u;
    if (j == n) a[1] += 1u;
    else if (j > n) a[2] += 1u;
    else a[3] += 1u;
    a[4] += steps;
    if (a[4] >= kFlushAt) flush();
  }
  if (tl >= 0) flush();
  __syncthreads();
  for (int i = threadIdx.x; i < n_tasks * kFields; i += blockDim.x) {
    const unsigned long long v =
        (unsigned long long)s_tally[2 * i] | ((unsigned long long)s_tally[2 * i + 1] << 32);
    if (v) atomicAdd(tally + i, v);
  }
}

}  // namespace

cudaError_t launch_inelastic_walk(const TaskDesc* d_tasks, int n_tasks, const EnergyDesc* d_edesc,
                                  const uint64_t* d_tab, const uint64_t* d_mode_tab,
                                  const double* d_c, const uint64_t* d_etab, int start_lead,
                                  uint64_t seed, uint64_t walkers_per_task, uint64_t id_offset,
                                  uint32_t max_steps, uint64_t* d_tally, int sm_count,
                                  cudaStream_t s) {
  if (n_tasks <= 0 || walkers_per_task == 0) return cudaSuccess;
  const PhiloxKey key{(uint32_t)seed, (uint32_t)(seed >> 32)};
  for (int w0 = 0; w0 < n_tasks; w0 += kWindow) {
    const int nt = (n_tasks - w0) < kWindow ? (n_tasks - w0) : kWindow;
    const size_t smem = sizeof(unsigned) * 2 * (size_t)nt * kFields;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, inelastic_walk_kernel,
                                                                  kThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const unsigned long long total = (unsigned long long)nt * walkers_per_task;
    unsigned long long blocks = (unsigned long long)sm_count * per_sm;
    const unsigned long long need = (total + kThreads - 1) / kThreads;
    if (blocks > need) blocks = need;
    inelastic_walk_kernel<<<(unsigned)blocks, kThreads, smem, s>>>(
        d_tasks, w0, nt, d_edesc, d_tab, d_mode_tab, d_c, d_etab, start_lead, key,
        walkers_per_task, id_offset, max_steps,
        reinterpret_cast<unsigned long long*>(d_tally) + (size_t)w0 * kFields,
        walk_chunk(total, blocks * (kThreads / 32)));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace negf
