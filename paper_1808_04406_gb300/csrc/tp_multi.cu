// Several steps per launch (multi_step.cuh) for the tensor-product lattices with
// FP32 storage and even nx.  us a step in chained launches and here, calls of 20 steps (3D)
// and 100: D3Q27 128^3 68.2 and 59.3, 256^3 524 and 479, D2Q9 2048^2 45.4 and 38.7, 4096^2 176
// and 125.  16-bit storage does not gain (D3Q27
// 256^3 FP16: 356 with the plane-walking sweep, 451 here; D2Q9 4096^2 BF16 119 and
// 152), nor does FP64, which its arithmetic binds (D2Q9 2048^2 854 and 958), nor odd
// nx (241 x 200 x 200 322 with column pairs, 377 here), nor the 37-velocity lattices, whose code for both parities exceeds the instruction cache
// (thermal FP16 1024^2 29.4 and 73).
#include "multi_step.cuh"
#include "sweep_body.cuh"

namespace lbm {
namespace {

struct TpGrid {
  tp::Grid g;
  Rates r;
  void* f;
  RowLength row;    // node pairs
  int unit_blocks;  // 2D: blocks of nodes per unit (a unit in 3D is a plane)
};

// Thread q of the unit's (3D) or the grid's (2D) run of pairs; false past its end.
template <int D>
__device__ __forceinline__ bool locate(const TpGrid& p, int unit, int block, int tid, int threads, int& i, int& y, int& z) {
  const uint32_t b = D == 3 ? (uint32_t)block : (uint32_t)unit * (uint32_t)p.unit_blocks + (uint32_t)block;
  z = D == 3 ? unit : 0;
  return row_of(b * (uint32_t)threads + (uint32_t)tid, p.row, p.g.ny, i, y);
}

template <int D>
struct PairUp {
  static constexpr int kThreads = 128, kMinBlocks = 4;
  using Params = TpGrid;
  static __device__ __forceinline__ bool update(bool odd, const TpGrid& p, int unit, int block, int tid) {
    return odd ? step<true>(p, unit, block, tid) : step<false>(p, unit, block, tid);
  }
  template <bool ODD>
  static __device__ __forceinline__ bool step(const TpGrid& p, int unit, int block, int tid) {
    int xp, y, z;
    if (!locate<D>(p, unit, block, tid, kThreads, xp, y, z)) return true;
    auto* f = static_cast<float*>(p.f);
    RawPair raw[tp::qof<D>()];
    tp::pair_load_raw<D, LBM_F32, ODD>(f, p.g, tp::PairAddr<D, ODD>(p.g, xp, y, z), raw);
    f2 om[2 * D + 1], v[tp::qof<D>()];
#pragma unroll
    for (int n = 0; n <= 2 * D; ++n) om[n] = cst<f2>(p.r.w[n]);
    tp::pair_decode<D, LBM_F32, ODD>(raw, v);
    // the stores' addresses are computed anew: kept from the loads they would take 54 registers
    if constexpr (D == 3) forget(xp, y, z);
    const bool ok = tp::collide<f2, D>(v, om);
    tp::pair_store<D, LBM_F32, ODD>(f, p.g, tp::PairAddr<D, ODD>(p.g, xp, y, z), v);
    return ok;
  }
};

template <typename Up>
cudaError_t run(Sim* s, int64_t n, const StepsCall& call, int* done) {
  const int64_t per_row = s->nx / 2;
  const int64_t plane_blocks = (s->ny * per_row + Up::kThreads - 1) / Up::kThreads;
  if (plane_blocks * Up::kThreads >= (int64_t)1 << 32) return cudaSuccess;
  const double bytes = (double)s->N * s->Q * (double)storage_elem_bytes(s->storage);
  const int blocks = multi_resident_blocks<Up>(s->stream);
  MultiPlan plan;
  // 2D: a node reaches the rows above and below, anywhere along them (periodic in x)
  multi_plan(n, s->D == 3 ? s->nz : 0, plane_blocks, 2.0 * per_row / Up::kThreads, bytes, blocks, (int)(s->step & 1),
             call.any_size, &plan);
  if (plan.steps < 2) return cudaSuccess;
  if (!call.launch) {
    *done = plan.steps;
    return cudaSuccess;
  }
  TpGrid p;
  p.g = tp::Grid{(int)s->nx, (int)s->ny, (int)s->nz, s->N};
  p.r = s->rates;
  p.f = s->pop;
  p.row = row_length(per_row);
  p.unit_blocks = plan.sub;
  const cudaError_t e = multi_launch<Up>(s, p, plan, blocks, call);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();  // not enough SMs for this stream: single sweeps need none
    return cudaSuccess;
  }
  if (e == cudaSuccess) *done = plan.steps;
  return e;
}

}  // namespace

cudaError_t tp_launch_steps(Sim* s, int64_t n, const StepsCall& call, int* done) {
  *done = 0;
  if (s->storage != LBM_F32 || !tp_pair_supported(s)) return cudaSuccess;
  return s->D == 2 ? run<PairUp<2>>(s, n, call, done) : run<PairUp<3>>(s, n, call, done);
}

}  // namespace lbm
