// Several time steps of a sweep in one cooperative launch, for grids larger than
// L2: a step only couples neighbouring rows (2D) or planes (3D), so step s + 1 can
// follow step s through the grid a little behind it, while what step s wrote is
// still in L2, and HBM sees the populations once for all of the steps.
//
// The grid is cut into units: planes of `tiles` thread blocks' work each in 3D, runs
// of consecutive nodes (one tile) in 2D.  Every resident block walks the tiles of
// all steps in one fixed order, block b taking entries b, b + G, b + 2 G, ...:
// iteration k holds, for every step s, the unit at position k - lag * s.
//
// Step s of unit u needs step s - 1 of units u - reach .. u + reach (AA slots belong
// to one node per step, so that is also all that may not be overwritten early).
// One counter per unit counts its finished tiles; a tile waits until those
// counters reach s * tiles.  All waits point to earlier entries of the order and
// all blocks are co-resident (cooperative launch), so the lowest unfinished tile
// can always run; each wait is bounded all the same.  A wait that gives up sets bit 2
// of the status word, and a word of this launch's own that ends the other waits (the
// status word's bit may be left from an earlier launch, and this one be sound).
//
// Step s starts at position s * reach instead of 0 (units taken modulo the grid),
// so that the periodic neighbours of its first unit have been finished by step
// s - 1.
//
// A tile is `sub` blocks of nodes one after the other: its completion costs a
// fence, of which an SM does one at a time in ~0.3 us.
#pragma once

#include <cuda.h>

#include "flat_index.cuh"
#include "lbm_internal.cuh"

namespace lbm {

struct MultiPlan {
  int units, tiles, steps;  // tiles: thread blocks' work per unit
  int sub;                  // blocks of nodes per tile
  int lag;                  // units between consecutive steps
  int reach;                // units that a node's velocities can reach on either side
  int first_odd;            // parity of the first step
  int outer;                // iterations
  int d_outer, d_mid, d_inner;  // the grid size as a step in (outer, mid, inner)
};

// They sit where reductions keep partials, behind the word that says a wait has given up.
constexpr int kMultiCounters = kRedBlocks * 8 * (int)sizeof(double) / 4 - 1;

__device__ __forceinline__ int load_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void add_release(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Up::update(odd, params, unit, block of nodes, thread): updates one node (or pair).
//
// One acquire (warp 0 looks at the counters of the next tile when it has finished
// this one), one barrier and one release per block and tile.  Warps that look and
// publish for themselves are far slower (0.5x on 256^3): fences and acquires, not
// the barrier, are what is scarce.
template <typename Up>
__global__ void __launch_bounds__(Up::kThreads, Up::kMinBlocks)
    multi_step_kernel(const __grid_constant__ typename Up::Params prm, const __grid_constant__ MultiPlan plan,
                      int* __restrict__ gave_up, int* __restrict__ status, int poll_limit) {
  int* const counters = gave_up + 1;
  __shared__ int ready[2];
  const int tid = threadIdx.x, mids = plan.steps;
  // the block's first entry
  int inner = blockIdx.x;
  int mid = inner / plan.tiles;
  inner -= mid * plan.tiles;
  int outer = mid / mids;
  mid -= outer * mids;
  auto advance = [&] {
    inner += plan.d_inner;
    if (inner >= plan.tiles) inner -= plan.tiles, ++mid;
    mid += plan.d_mid;
    if (mid >= mids) mid -= mids, ++outer;
    outer += plan.d_outer;
  };
  // the step and unit of the entry, skipping those outside the step's positions
  auto next_entry = [&](int& s, int& u) {
    for (; outer < plan.outer; advance()) {
      s = mid;
      const int p = outer - plan.lag * s, first = s * plan.reach;
      u = p >= plan.units ? p - plan.units : p;
      if (p >= first && p < plan.units + first) return true;
    }
    return false;
  };
  // the lanes of warp 0 look at the counters that (s, u) waits for
  auto satisfied = [&](int s, int u) -> int {
    int ok = 1;
    if (s > 0) {
      for (int j = tid; j <= 2 * plan.reach; j += 32) {
        int v = u + j - plan.reach;
        v = v < 0 ? v + plan.units : (v >= plan.units ? v - plan.units : v);
        if (load_acquire(counters + v) < s * plan.tiles) ok = 0;
      }
    }
    return __all_sync(0xffffffffu, ok);
  };

  int s, u, buf = 0;
  bool more = next_entry(s, u);
  bool known = s == 0;  // the tile's inputs are known to be complete (the same in every thread)
  while (more) {
    if (!known) {
      int give_up = 0;
      if (tid < 32) {
        int polls = 0;
        while (!satisfied(s, u)) {
          // the whole warp or none of it: satisfied() takes all lanes
          if (++polls > poll_limit || (polls % 1024 == 0 && __any_sync(0xffffffffu, load_acquire(gave_up) != 0))) {
            give_up = 1;
            break;
          }
        }
        if (give_up && tid == 0) {
          atomicOr(status, 2);
          atomicExch(gave_up, 1);
        }
      }
      if (__syncthreads_or(give_up)) return;
    }
    const int t = inner;
    int s1 = 0, u1 = 0;
    advance();
    const bool more1 = next_entry(s1, u1);
    bool ok = true;
    const bool odd = ((plan.first_odd + s) & 1) != 0;
    for (int k = 0; k < plan.sub; ++k) ok = Up::update(odd, prm, u, t * plan.sub + k, tid) && ok;
    if (!ok) atomicOr(status, 1);
    if (tid < 32 && more1) {
      const int r = satisfied(s1, u1);
      if (tid == 0) ready[buf] = r;
    }
    __syncthreads();  // the tile's stores have been issued, ready[buf] is written
    if (tid == Up::kThreads - 1 && s + 1 < plan.steps) add_release(counters + u, 1);
    known = more1 && ready[buf];
    buf ^= 1;
    more = more1;
    s = s1;
    u = u1;
  }
}

// Whether the stream's work may run on some of the device's SMs only.
inline bool multi_green_context(cudaStream_t stream) {
  using GetGreenCtx = CUresult (*)(CUstream, CUgreenCtx*);
  static const GetGreenCtx get = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuStreamGetGreenCtx", &p, 12040, cudaEnableDefault, &found);
    return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? reinterpret_cast<GetGreenCtx>(p) : nullptr;
  }();
  CUgreenCtx green = nullptr;
  return get && get(stream, &green) == CUDA_SUCCESS && green != nullptr;
}

// Blocks of the kernel that are resident at once on the current device for work of this
// stream, 0 if that is not known: in a green context, which has fewer SMs, a launch that
// counts on all of them would be refused.
template <typename Up>
int multi_resident_blocks(cudaStream_t stream) {
  int dev = 0, sms = 0, per = 0;
  if (multi_green_context(stream) || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, multi_step_kernel<Up>, Up::kThreads, 0) != cudaSuccess)
    return 0;
  return sms * per;
}

// How much of the 129 MB L2 the populations between the first and the last step may
// take (D3Q27 FP32 256^3: 476 us a step with 64 MB, 486 with 90), and the size up to
// which a whole grid stays in L2 by itself.  us a step in chained launches and here,
// D3Q27: 96^3 (96 MB) 26.8 and 28.1, 100^3 (108 MB) 32.3 and 38.5, 104^3 (121 MB) 37.9
// and 36.7, 108^3 (136 MB) 43.3 and 41.7, 128^3 68.2 and 59.3, 160^3 131.8 and 114.6, 192^3
// 222 and 197, 256^3 524 and 479, 320^3 1023 and 965; D2Q9: 1600^2 (92 MB) 22.1 and 25.5,
// 1900^2 (130 MB) 39.7 and 36.1, 2048^2 45.4 and 38.7.
constexpr int64_t kMultiBytes = (int64_t)64 << 20;
constexpr int64_t kResidentBytes = (int64_t)128 << 20;
constexpr int kMultiMaxReach = 63;
// Blocks of nodes per tile at most: more put the steps further apart (256^3: 504,
// 476 and 525 us a step with 1, 2 and 4), fewer cost fences.
constexpr int kMultiMaxSub = 2;
// Steps per launch at most.  A launch holds every block slot of the GPU until its last
// step, and L2 has room for many steps of a 2D grid or of small planes (4096 x 1801: 85
// of 170 steps, 6.5 ms a launch; 256^3 has 3, 1.4 ms).  us a step in calls of 100 steps,
// without a limit and so: D2Q9 2048^2 40.9 and 38.7, 4096^2 134.8 and 125.5, 4096 x 1801
// 76.3 and 73.5, D3Q27 32 x 32 x 2000 58.4 and 54.5, 66 x 50 x 400 42.3 and 41.6.
constexpr int kMultiMaxSteps = 32;

// Plan of up to n steps over `planes` planes of `plane_blocks` blocks of nodes (3D),
// or over one run of plane_blocks blocks (planes = 0, 2D) whose velocities reach
// `reach_blocks` blocks (rounded up) on either side; `bytes` of populations in all
// and G resident blocks.  any_size: also where the whole grid stays in L2.
// plan->steps < 2 where several steps at a time are not possible.
inline void multi_plan(int64_t n, int64_t planes, int64_t plane_blocks, double reach_blocks, double bytes, int G,
                       int first_odd, bool any_size, MultiPlan* plan) {
  plan->steps = 0;
  if (n < 2 || G < 1 || (bytes <= (double)kResidentBytes && !any_size)) return;
  const int64_t blocks = (planes ? planes : 1) * plane_blocks;
  // two tiles or more per block and step, so that waits overlap with work
  int64_t sub = blocks / (2 * G);
  sub = sub < 1 ? 1 : sub > kMultiMaxSub ? kMultiMaxSub : sub;
  if (sub > plane_blocks) sub = plane_blocks;
  int64_t units, tiles, reach;
  if (planes) {
    units = planes;
    tiles = (plane_blocks + sub - 1) / sub;
    reach = 1;
  } else {
    while ((blocks + sub - 1) / sub > kMultiCounters) ++sub;
    units = (blocks + sub - 1) / sub;
    tiles = 1;
    // one more across the periodic boundary, where the last unit may be short
    reach = (int64_t)(reach_blocks / (double)sub) + 2;
  }
  if (units > kMultiCounters || reach > kMultiMaxReach || 2 * reach + 1 > units) return;
  // far enough behind that a tile's inputs were dispatched more than a wave of blocks ago
  const double unit_bytes = bytes / (double)units;
  auto lag_of = [&](int64_t T) { return reach + (5 * G / 4 + T * tiles - 1) / (T * tiles); };
  auto fits = [&](int64_t T) {
    return T * reach <= units && (double)(lag_of(T) * (T - 1) + 2 * reach + 1) * unit_bytes <= (double)kMultiBytes;
  };
  if (!fits(2)) return;
  int64_t T = 2;
  while (T < n && T < kMultiMaxSteps && fits(T + 1)) ++T;
  const int64_t passes = (n + T - 1) / T;  // equal passes
  n = (n + passes - 1) / passes;
  if (n < 2 || n * tiles >= ((int64_t)1 << 30) || units * tiles >= ((int64_t)1 << 30)) return;
  plan->lag = (int)lag_of(n);
  plan->units = (int)units;
  plan->tiles = (int)tiles;
  plan->sub = (int)sub;
  plan->reach = (int)reach;
  plan->steps = (int)n;
  plan->first_odd = first_odd;
  plan->outer = (int)(units + (plan->lag + reach) * (n - 1));
}

template <typename Up>
cudaError_t multi_launch(Sim* s, const typename Up::Params& prm, MultiPlan plan, int blocks, const StepsCall& call) {
  const int64_t G = blocks;
  plan.d_inner = (int)(G % plan.tiles);
  plan.d_mid = (int)(G / plan.tiles % plan.steps);
  plan.d_outer = (int)(G / plan.tiles / plan.steps);
  int* gave_up = reinterpret_cast<int*>(partials_buf(s));
  cudaError_t e = cudaMemsetAsync(gave_up, 0, (size_t)(1 + plan.units) * sizeof(int), s->stream);
  if (e == cudaSuccess && call.starve)  // large negative numbers
    e = cudaMemsetAsync(gave_up + 1, 0x80, (size_t)plan.units * sizeof(int), s->stream);
  if (e != cudaSuccess) return e;
  int* status = status_word(s);
  int polls = call.polls;
  typename Up::Params p = prm;
  void* args[] = {&p, &plan, &gave_up, &status, &polls};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(multi_step_kernel<Up>), dim3((unsigned)G),
                                     dim3(Up::kThreads), args, 0, s->stream);
}

}  // namespace lbm
