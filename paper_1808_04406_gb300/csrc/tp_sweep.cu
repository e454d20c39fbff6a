// Fused stream + collide sweep (one lattice Boltzmann time step) for the
// tensor-product lattices D2Q9 and D3Q27, in place with the AA pattern.
//
// One thread owns one node (or two of a column, tp_column_kernel).  Even sweep: read the node's own slots, collide,
// write each result into the opposite slot of the same node.  Odd sweep: read
// population opp(j) from slot (x + e_j, j), collide, write population j to the
// same slot (x + e_j, j).  Both read and write exactly Q values per node, so a
// step moves 2 Q sizeof(storage) bytes per node through HBM.
//
// The collision is the CM-MRT operator of Sec. II.C (Eq. omega, final update)
// evaluated per axis in registers: populations -> raw moments -> central
// moments -> relax order by order -> raw moments -> populations.
#include "flat_index.cuh"
#include "pdl.cuh"
#include "sweep_body.cuh"

namespace lbm {
namespace {

// Launch shape: threads per block along x, and the minimum resident blocks per
// SM requested from the register allocator.
#ifndef LBM_SWEEP_THREADS
#define LBM_SWEEP_THREADS 128
#endif
#ifndef LBM_SWEEP_MINB
#define LBM_SWEEP_MINB 1
#endif
constexpr int kSweepThreads = LBM_SWEEP_THREADS;

template <int D, int S, bool ODD>
__global__ void __launch_bounds__(kSweepThreads, LBM_SWEEP_MINB)
    tp_sweep_kernel(typename tp::Store<S>::type* __restrict__ f, tp::Grid g, Rates r,
                    int* __restrict__ status, RowLength row, int z0) {
  using T = typename tp::Store<S>::calc;
  int x, y;
  const bool in = row_of(blockIdx.x * blockDim.x + threadIdx.x, row, g.ny, x, y);
  const int z = blockIdx.z + z0;  // z0: first plane of the swept range
  chain_wait();
  if (!in) return;
  T om[2 * D + 1];
#pragma unroll
  for (int n = 0; n <= 2 * D; ++n) om[n] = (T)r.w[n];

  if (!tp::update_node<D, S, ODD>(f, g, om, x, y, z)) atomicOr(status, 1);
}

// Two nodes of one column, (x, y) and (x, y + 1), per thread in packed FP32x2, for
// 16/32-bit storage: odd nx leaves x-neighbour pairs unaligned, while a lane of
// each of two rows is read and written in 1-element accesses along x that
// coalesce.  Half the instructions of one node per thread.  On the last row of an
// odd ny, lane 1 repeats lane 0's node: both lanes load the same slots, compute
// the same values and store them twice to the same places.  Populations are those of
// one node per thread bit for bit (tests/test_gpu_odd_rows.py): which kernel a grid
// takes, or a slab of its planes, does not show.
// us a step with one node per thread and so: D3Q27 FP32 161 x 95 x 77 47.7 and 42.0,
// 241 x 200 x 200 369 and 322, FP16 129 x 128 x 128 69.7 and 57.1; D2Q9 BF16 1023^2 9.9
// and 9.3, but FP32 1023 x 1024 9.8 and 10.2.  Grids of less than a wave of blocks
// keep their nodes on twice the threads (33^3 3.2 and 4.0, 161 x 95 x 4 3.9 and 4.2).  In the
// second wave the two change over: FP32 53^3 (636 blocks) 6.4 and 7.6, 97 x 64 x 31 (775)
// 7.5 and 8.4, 65^3 (1105) 10.4 and 10.3, 161 x 95 x 20 (1220) 11.0 and 10.8.
template <int D, bool ODD>
struct ColumnPair {
  uint32_t xo[3], zo[3];
  uint32_t ro[2][3];  // row offsets of the lanes for e_y = -1, 0, +1
  __device__ __forceinline__ ColumnPair(const tp::Grid& g, int x, int y, int z) {
    const uint32_t nx = (uint32_t)g.nx, nxy = (uint32_t)g.nx * (uint32_t)g.ny;
    const int y1 = y + 1 < g.ny ? y + 1 : y;
    xo[1] = (uint32_t)x;
    ro[0][1] = nx * (uint32_t)y;
    ro[1][1] = nx * (uint32_t)y1;
    zo[0] = zo[1] = zo[2] = D == 3 ? nxy * (uint32_t)z : 0u;
    if (ODD) {
      xo[0] = (uint32_t)(x == 0 ? g.nx - 1 : x - 1);
      xo[2] = (uint32_t)(x == g.nx - 1 ? 0 : x + 1);
      ro[0][0] = nx * (uint32_t)(y == 0 ? g.ny - 1 : y - 1);
      ro[0][2] = nx * (uint32_t)(y == g.ny - 1 ? 0 : y + 1);
      ro[1][0] = nx * (uint32_t)(y1 == 0 ? g.ny - 1 : y1 - 1);
      ro[1][2] = nx * (uint32_t)(y1 == g.ny - 1 ? 0 : y1 + 1);
      if (D == 3) {
        zo[0] = nxy * (uint32_t)(z == 0 ? g.nz - 1 : z - 1);
        zo[2] = nxy * (uint32_t)(z == g.nz - 1 ? 0 : z + 1);
      }
    }
  }
  __device__ __forceinline__ uint32_t slot(int j, int lane) const {
    if (!ODD) return xo[1] + ro[lane][1] + zo[1];
    return xo[tp::dig(j, 0)] + ro[lane][tp::dig(j, 1)] + (D == 3 ? zo[tp::dig(j, 2)] : 0u);
  }
};

template <int D, int S, bool ODD>
__global__ void __launch_bounds__(kSweepThreads, D == 3 ? 4 : 6)
    tp_column_kernel(typename PairIO<S>::E* __restrict__ f, tp::Grid g, Rates r, int* __restrict__ status,
                     RowLength row, int z0) {
  using IO = PairIO<S>;
  int x, y;
  const bool in = row_of(blockIdx.x * blockDim.x + threadIdx.x, row, (g.ny + 1) >> 1, x, y);
  int z = blockIdx.z + z0;  // z0: first plane of the swept range
  chain_wait();
  if (!in) return;
  y *= 2;
  f2 om[2 * D + 1], v[tp::qof<D>()];
#pragma unroll
  for (int n = 0; n <= 2 * D; ++n) om[n] = cst<f2>(r.w[n]);
  {
    const ColumnPair<D, ODD> A(g, x, y, z);
    RawPair raw[tp::qof<D>()];
#pragma unroll
    for (int j = 0; j < tp::qof<D>(); ++j) {
      const auto* fj = f + (size_t)j * g.N;
      IO::raw11(fj + A.slot(j, 0), fj + A.slot(j, 1), raw[j]);
    }
#pragma unroll
    for (int j = 0; j < tp::qof<D>(); ++j) {
      f2 val = IO::dec11(raw[j]);
      if (IO::kScaled) val = val * cst<f2>(tp::wq<D>(j));
      v[ODD ? tp::opp<D>(j) : j] = val;
    }
  }
  // the stores' addresses are computed anew: kept from the loads they would take too many registers
  forget(x, y, z);
  if (!tp::collide<f2, D, false, D == 2>(v, om)) atomicOr(status, 1);
  const ColumnPair<D, ODD> A(g, x, y, z);
#pragma unroll
  for (int j = 0; j < tp::qof<D>(); ++j) {
    auto* fj = f + (size_t)j * g.N;
    f2 val = ODD ? v[j] : v[tp::opp<D>(j)];
    if (IO::kScaled) val = val * cst<f2>(tp::iwq<D>(j));
    IO::store11(fj + A.slot(j, 0), fj + A.slot(j, 1), val);
  }
}

inline int64_t column_blocks(const Sim* s) { return (s->nx * ((s->ny + 1) / 2) + kSweepThreads - 1) / kSweepThreads; }
// Whether the sweep takes node pairs of a column (see above).
inline bool columns(const Sim* s) {
  return s->storage != LBM_F64 && !(s->D == 2 && s->storage == LBM_F32) && column_blocks(s) * active_nz(s) >= 4 * 152;
}

template <int D, int S>
cudaError_t launch_columns(Sim* s, int odd) {
  tp::Grid g{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  dim3 grid((unsigned)column_blocks(s), 1, (unsigned)active_nz(s));
  return launch_chained(odd ? tp_column_kernel<D, S, true> : tp_column_kernel<D, S, false>, grid, dim3(kSweepThreads), 0,
                        s->stream, static_cast<typename PairIO<S>::E*>(s->pop), g, s->rates, status_word(s),
                        row_length(s->nx), (int)active_z0(s));
}

template <int D, int S>
cudaError_t launch(Sim* s, int odd) {
  using Tst = typename tp::Store<S>::type;
  tp::Grid g{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  dim3 block(kSweepThreads);
  dim3 grid((unsigned)((s->nx * s->ny + kSweepThreads - 1) / kSweepThreads), 1, (unsigned)active_nz(s));
  Tst* f = static_cast<Tst*>(s->pop);
  const int z0 = (int)active_z0(s);
  return launch_chained(odd ? tp_sweep_kernel<D, S, true> : tp_sweep_kernel<D, S, false>, grid, block, 0, s->stream, f, g,
                        s->rates, status_word(s), row_length(s->nx), z0);
}

template <int D>
cudaError_t launch_d(Sim* s, int odd) {
  switch (s->storage) {
    case LBM_F64: return launch<D, LBM_F64>(s, odd);
    case LBM_F32:
      if (D == 3 && columns(s)) return launch_columns<3, LBM_F32>(s, odd);
      return launch<D, LBM_F32>(s, odd);
    case LBM_F16: return columns(s) ? launch_columns<D, LBM_F16>(s, odd) : launch<D, LBM_F16>(s, odd);
    case LBM_BF16: return columns(s) ? launch_columns<D, LBM_BF16>(s, odd) : launch<D, LBM_BF16>(s, odd);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

const char* tp_sweep_kernel_name(const Sim* s) { return columns(s) ? "tp_column_kernel" : "tp_sweep_kernel"; }

cudaError_t tp_launch_sweep(Sim* s, int odd) {
  return s->D == 2 ? launch_d<2>(s, odd) : launch_d<3>(s, odd);
}

}  // namespace lbm
