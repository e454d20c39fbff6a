// Fused stream + collide sweep, two neighbouring nodes (x0, x0 + 1) per thread,
// for FP32 / FP16 / BF16 offset storage on D2Q9 and D3Q27 (nx even).
//
// Same AA pattern and collision as the one-node sweep (tp_sweep.cu); the two
// nodes' values for one population sit in the two lanes of a packed FP32x2
// register, so every arithmetic instruction advances both nodes.
//
// Pairing.  The even sweep reads and writes the nodes' own slots, so it pairs
// (x0, x0 + 1) with x0 even and every access is one aligned 2-element access.
// The odd sweep touches slots shifted by e_x; it pairs (x0, x0 + 1 mod nx) with
// x0 odd, so that the shifted slots of e_x = -1 (x0 - 1, x0) and of e_x = +1
// (x0 + 1, x0 + 2, mod nx) start at an even x and stay aligned; only the nine
// populations with e_x = 0 need two 1-element accesses.  The last odd pair
// (nx - 1, 0) wraps around the row.
//
// D3Q27 with 16-bit offsets runs tp_pair_zrun_kernel: the same pairs, each
// thread walking several planes with the next plane's loads in flight.
#include <cstdlib>
#include <cstring>

#include "flat_index.cuh"
#include "pdl.cuh"
#include "sweep_body.cuh"

namespace lbm {
namespace {

#ifndef LBM_PAIR_THREADS
#define LBM_PAIR_THREADS 128
#endif
constexpr int kPairThreads = LBM_PAIR_THREADS;
// Blocks per SM: with the stores' addresses computed anew instead of kept from the
// loads (54 registers on D3Q27) the sweeps take 128 registers or less.
constexpr int kPairMinBlocks = 4;

template <int D, int S, bool ODD>
__global__ void __launch_bounds__(kPairThreads, kPairMinBlocks)
    tp_pair_kernel(typename PairIO<S>::E* __restrict__ f, tp::Grid g, Rates r,
                   int* __restrict__ status, RowLength row, int z0) {
  int xp, y;
  const bool in = row_of(blockIdx.x * blockDim.x + threadIdx.x, row, g.ny, xp, y);
  int z = blockIdx.z + z0;  // z0: first plane of the swept range
  chain_wait();
  if (!in) return;
  f2 om[2 * D + 1];
#pragma unroll
  for (int n = 0; n <= 2 * D; ++n) om[n] = cst<f2>(r.w[n]);
  f2 v[tp::qof<D>()];
  tp::pair_load<D, S, ODD>(f, g, tp::PairAddr<D, ODD>(g, xp, y, z), v);
  if constexpr (D == 3) forget(xp, y, z);
  if (!tp::collide<f2, D>(v, om)) atomicOr(status, 1);
  tp::pair_store<D, S, ODD>(f, g, tp::PairAddr<D, ODD>(g, xp, y, z), v);
}

// The same sweep for D3Q27 with 16-bit offsets, each thread walking kZRun
// consecutive planes of its pair column (x0, x0 + 1, y): the raw 16-bit words
// of the next plane's pair are loaded before the current pair is decoded and
// collided, so their latency overlaps the collision instead of stalling it.
// (AA slots belong to one node per sweep, so loading the next pair before the
// current one is stored is race-free.)  The node arithmetic is that of
// tp_pair_kernel, and so are the results, bit for bit.  At 4 blocks per SM
// the compiler keeps it within 128 registers (16 bytes spilled in the odd sweep, which
// executes 1112 instructions per pair against the even one's 782: addresses of shifted
// slots, and 2-byte accesses for e_x = 0).
//
// The walk is 8 planes, or fewer where that would leave less than 900 blocks, one
// and a half waves of 608 (FP16, us a step, walks of 8 and of 1: 64^3 10.9 and 7.7,
// 96^3 28.5 and 21.2, 128^3 with 1024 blocks 49.8 and 51.9, 256^3 356 and 401).
constexpr int kZRun = 8;
constexpr int kZRunMinBlocks = 4;
constexpr int kZRunMinGrid = 900;

template <int S, bool ODD>
__global__ void __launch_bounds__(kPairThreads, kZRunMinBlocks)
    tp_pair_zrun_kernel(typename PairIO<S>::E* __restrict__ f, tp::Grid g, Rates r, int* __restrict__ status,
                        RowLength row, int z0, int z1, int run) {
  int xp, y;
  const bool in = row_of(blockIdx.x * blockDim.x + threadIdx.x, row, g.ny, xp, y);
  chain_wait();
  if (!in) return;
  const int zb = z0 + (int)blockIdx.z * run;
  const int ze = zb + run < z1 ? zb + run : z1;  // planes zb .. ze - 1
  f2 om[7];
#pragma unroll
  for (int n = 0; n < 7; ++n) om[n] = cst<f2>(r.w[n]);
  RawPair raw[27];
  tp::pair_load_raw<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, zb), raw);
  bool ok = true;
  for (int z = zb; z < ze; ++z) {
    f2 v[27];
    tp::pair_decode<3, S, ODD>(raw, v);
    if (z + 1 < ze) tp::pair_load_raw<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, z + 1), raw);
    ok = tp::collide<f2, 3>(v, om) && ok;
    int zs = z;
    forget(xp, y, zs);
    tp::pair_store<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, zs), v);
  }
  if (!ok) atomicOr(status, 1);
}

// The five sums of a warp, each by the tree of offsets 16, 8, 4, 2, 1.  Where two values
// are left to reduce, the halves of the warp take one each (addition commutes, so every
// sum is that of the five separate trees, bit for bit): 8 shuffles instead of 25.
// A D3Q27 FP32 run of 20 steps with totals on 128^3, fields in and out: 2636 us with 25
// shuffles in plain launches at 3 blocks per SM, 2186 so.  (One tree for 4 planes of a
// thread takes 2062, but other nodes of a warp meet in FP32: totals 2e-8 apart.)
__device__ __forceinline__ float fold2(float a, float b, int o, int lane) {
  const bool up = (lane & o) != 0;
  return (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, o);
}
__device__ __forceinline__ float fold1(float a, int o) { return a + __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ void write_partials(const float (&acc)[5], float* __restrict__ partials) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float s = fold2(fold2(acc[0], acc[1], 16, lane), fold2(acc[2], acc[3], 16, lane), 8, lane);
  s = fold2(s, fold1(fold1(acc[4], 16), 8), 4, lane);
  s = fold1(fold1(s, 2), 1);
  // sum k now sits in lane 0, 16, 8, 24, 4
  const int k = lane & 4 ? 4 : (lane >> 4) + ((lane & 8) >> 2);
  if ((lane & 3) == 0 && (k < 4 || lane == 4)) {
    const size_t b = (size_t)blockIdx.x + (size_t)gridDim.x * ((size_t)blockIdx.y + (size_t)gridDim.y * blockIdx.z);
    partials[(b * (kPairThreads / 32) + (size_t)wid) * 8 + k] = s;
  }
}

// The plane-walking sweep with the totals of the consumed state, as
// tp_pair_totals_kernel computes them per node; each thread adds its nodes of
// all its planes in FP32 before the warp's shuffle tree, so there is one
// partial per warp of this grid (tp_pair_warps).  Walks of kZRun planes on every grid,
// and threads along the rows (see tp_pair_totals_kernel).
template <int S, bool ODD>
__global__ void __launch_bounds__(kPairThreads, 3)  // the running totals need more than 128 registers
    tp_pair_zrun_totals_kernel(typename PairIO<S>::E* __restrict__ f, tp::Grid g, Rates r,
                               int* __restrict__ status, float* __restrict__ partials, int z0, int z1) {
  const int xp = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  float acc[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  chain_wait();
  if (xp < (g.nx >> 1)) {
    const int zb = z0 + (int)blockIdx.z * kZRun;
    const int ze = zb + kZRun < z1 ? zb + kZRun : z1;
    f2 om[7];
#pragma unroll
    for (int n = 0; n < 7; ++n) om[n] = cst<f2>(r.w[n]);
    RawPair raw[27];
    tp::pair_load_raw<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, zb), raw);
    bool ok = true;
    for (int z = zb; z < ze; ++z) {
      f2 v[27];
      tp::pair_decode<3, S, ODD>(raw, v);
      if (z + 1 < ze) tp::pair_load_raw<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, z + 1), raw);
      tp::NodeMoments<f2, 3> m;
      ok = tp::collide<f2, 3, true>(v, om, &m) && ok;
      tp::pair_store<3, S, ODD>(f, g, tp::PairAddr<3, ODD>(g, xp, y, z), v);
      float d0, d1, jj0 = 0.0f, jj1 = 0.0f;
      unpack2(m.drho, d0, d1);
      acc[0] += d0 + d1;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        float j0, j1;
        unpack2(m.j[d], j0, j1);
        acc[1 + d] += j0 + j1;
        jj0 += j0 * j0;
        jj1 += j1 * j1;
      }
      acc[4] += __fdividef(0.5f * jj0, 1.0f + d0) + __fdividef(0.5f * jj1, 1.0f + d1);
    }
    if (!ok) atomicOr(status, 1);
  }
  write_partials(acc, partials);
}

// The same sweep, which also writes per block the FP64 totals of the state it
// consumed: sum (rho - 1), sum rho u_d, sum rho |u|^2 / 2 (as the grid
// reduction defines them, per node from the collision's own moments) to
// partials[warp * 8 + k] (FP32), one entry per warp of the grid.  A warp sums
// its 64 nodes in FP32 (a fixed shuffle tree); the warps' sums are added in
// FP64 afterwards.  (FP64 arithmetic runs at a small fraction of the FP32 rate on
// this GPU: per-node FP64 sums would double the sweep's time; and no block
// barrier holds finished warps back.)
//
// Threads run along the rows here, and a warp's 64 nodes are of one row: which nodes a
// warp adds up in FP32 decides the last bits of the totals.
template <int D, int S, bool ODD>
__global__ void __launch_bounds__(kPairThreads, kPairMinBlocks)
    tp_pair_totals_kernel(typename PairIO<S>::E* __restrict__ f, tp::Grid g, Rates r, int* __restrict__ status,
                          float* __restrict__ partials, int z0) {
  int xp = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z + z0;
  float acc[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  chain_wait();
  if (xp < (g.nx >> 1)) {
    f2 om[2 * D + 1];
#pragma unroll
    for (int n = 0; n <= 2 * D; ++n) om[n] = cst<f2>(r.w[n]);
    f2 v[tp::qof<D>()];
    tp::pair_load<D, S, ODD>(f, g, tp::PairAddr<D, ODD>(g, xp, y, z), v);
    if constexpr (D == 3) forget(xp, y, z);
    tp::NodeMoments<f2, D> m;
    const bool ok = tp::collide<f2, D, true>(v, om, &m);
    tp::pair_store<D, S, ODD>(f, g, tp::PairAddr<D, ODD>(g, xp, y, z), v);
    if (!ok) atomicOr(status, 1);
    float d0, d1, jj0 = 0.0f, jj1 = 0.0f;
    unpack2(m.drho, d0, d1);
    acc[0] = d0 + d1;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      float j0, j1;
      unpack2(m.j[d], j0, j1);
      acc[1 + d] = j0 + j1;
      jj0 += j0 * j0;
      jj1 += j1 * j1;
    }
    acc[4] = __fdividef(0.5f * jj0, 1.0f + d0) + __fdividef(0.5f * jj1, 1.0f + d1);
  }
  write_partials(acc, partials);
}

// LBM_TP_ZRUN=0 keeps one pair per thread for 16-bit D3Q27 (read at every
// launch; used to compare the two kernels).
bool zrun_enabled() {
  const char* e = std::getenv("LBM_TP_ZRUN");
  return !(e && std::strcmp(e, "0") == 0);
}

inline unsigned plane_blocks(const Sim* s) {
  return (unsigned)((s->nx / 2 * s->ny + kPairThreads - 1) / kPairThreads);
}

// Planes per thread.
inline int walk_of(const Sim* s) {
  int run = kZRun;
  while (run > 1 && (int64_t)plane_blocks(s) * ((active_nz(s) + run - 1) / run) < kZRunMinGrid) run /= 2;
  return run;
}

template <int S>
cudaError_t launch_zrun(Sim* s, int odd) {
  using E = typename PairIO<S>::E;
  tp::Grid g{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  const int64_t nzs = active_nz(s);
  const int run = walk_of(s);
  dim3 grid(plane_blocks(s), 1, (unsigned)((nzs + run - 1) / run));
  const int z0 = (int)active_z0(s), z1 = (int)(active_z0(s) + nzs);
  E* f = static_cast<E*>(s->pop);
  return launch_chained(odd ? tp_pair_zrun_kernel<S, true> : tp_pair_zrun_kernel<S, false>, grid, dim3(kPairThreads), 0,
                        s->stream, f, g, s->rates, status_word(s), row_length(s->nx / 2), z0, z1, run);
}

template <int D, int S>
cudaError_t launch(Sim* s, int odd) {
  using E = typename PairIO<S>::E;
  if constexpr (D == 3 && S != LBM_F32) {
    if (zrun_enabled()) return launch_zrun<S>(s, odd);
  }
  tp::Grid g{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  dim3 block(kPairThreads);
  dim3 grid(plane_blocks(s), 1, (unsigned)active_nz(s));
  const int z0 = (int)active_z0(s);
  E* f = static_cast<E*>(s->pop);
  return launch_chained(odd ? tp_pair_kernel<D, S, true> : tp_pair_kernel<D, S, false>, grid, block, 0, s->stream, f, g,
                        s->rates, status_word(s), row_length(s->nx / 2), z0);
}

// blocks of the totals sweeps: rows, each of one or more blocks, and planes or walks of kZRun
inline dim3 totals_grid(const Sim* s) {
  const int64_t run = s->D == 3 && s->storage != LBM_F32 && zrun_enabled() ? kZRun : 1;
  return dim3((unsigned)((s->nx / 2 + kPairThreads - 1) / kPairThreads), (unsigned)s->ny,
              (unsigned)((active_nz(s) + run - 1) / run));
}

template <int D, int S>
cudaError_t launch_totals(Sim* s, int odd, float* partials) {
  using E = typename PairIO<S>::E;
  tp::Grid g{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  const int z0 = (int)active_z0(s), z1 = (int)(z0 + active_nz(s));
  E* f = static_cast<E*>(s->pop);
  if constexpr (D == 3 && S != LBM_F32) {
    if (zrun_enabled())
      return launch_chained(odd ? tp_pair_zrun_totals_kernel<S, true> : tp_pair_zrun_totals_kernel<S, false>,
                            totals_grid(s), dim3(kPairThreads), 0, s->stream, f, g, s->rates, status_word(s), partials,
                            z0, z1);
  }
  return launch_chained(odd ? tp_pair_totals_kernel<D, S, true> : tp_pair_totals_kernel<D, S, false>, totals_grid(s),
                        dim3(kPairThreads), 0, s->stream, f, g, s->rates, status_word(s), partials, z0);
}

template <int D>
cudaError_t launch_totals_d(Sim* s, int odd, float* partials) {
  switch (s->storage) {
    case LBM_F32: return launch_totals<D, LBM_F32>(s, odd, partials);
    case LBM_F16: return launch_totals<D, LBM_F16>(s, odd, partials);
    case LBM_BF16: return launch_totals<D, LBM_BF16>(s, odd, partials);
  }
  return cudaErrorInvalidValue;
}

template <int D>
cudaError_t launch_d(Sim* s, int odd) {
  switch (s->storage) {
    case LBM_F32: return launch<D, LBM_F32>(s, odd);
    case LBM_F16: return launch<D, LBM_F16>(s, odd);
    case LBM_BF16: return launch<D, LBM_BF16>(s, odd);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool tp_pair_supported(const Sim* s) { return s->storage != LBM_F64 && (s->nx % 2) == 0; }

const char* tp_pair_kernel_name(const Sim* s) {
  return s->D == 3 && s->storage != LBM_F32 && zrun_enabled() ? "tp_pair_zrun_kernel" : "tp_pair_kernel";
}

cudaError_t tp_launch_pair_sweep(Sim* s, int odd) {
  return s->D == 2 ? launch_d<2>(s, odd) : launch_d<3>(s, odd);
}

int64_t tp_pair_warps(const Sim* s) {
  const dim3 b = totals_grid(s);
  return (int64_t)b.x * b.y * b.z * (kPairThreads / 32);
}

cudaError_t tp_launch_pair_sweep_totals(Sim* s, int odd, float* partials) {
  return s->D == 2 ? launch_totals_d<2>(s, odd, partials) : launch_totals_d<3>(s, odd, partials);
}

}  // namespace lbm
