// step_f16sr.cu -- the F16S form (FP16 of 1024 (f - w rho0), the shifted
// storage of the populations) stepped with stochastically rounded stores.
//
// Round-to-nearest FP16 drops every per-step change below half an ulp of the
// stored value, and near a steady state those are all of them: the stored
// state freezes short of the steady state at the same nodes every step.
// Stochastic rounding keeps such changes on average (see sround.cuh).  The
// stored layout, decoding and collision are those of the F16S step kernel;
// only the store differs, so state import and export, fields and every
// other entry point treat the lattice as F16S.
#include "kernels.cuh"
#include "sround.cuh"
#include "launch_f16sr.h"

namespace clbm {
namespace {

// One node per thread.
template <bool FORCE, bool CHECK, bool UNIT>
__global__ void __launch_bounds__(256) step_sr_kernel(const StepArgs<__half, float> a,
                                                      const StepSeed seed) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = a.zrev ? a.nz - 1 - int(blockIdx.z) : int(blockIdx.z);
  const bool active = x < a.nx && y < a.ny;
  if (!CHECK && !active) return;
  CheckSums sums;
  if (active) {
    const int i = z * a.plane + y * a.pitch + x;
    float d[Q];
    pull_node(a, x, y, z, i, d);
    NodeOut<float> o;
    collide<float, FORCE, pair_out<__half>(), log2_scale<__half>(), UNIT>(a.C, d, o);
    // the deviations are carried scaled by 1024, as they are stored
    store_sr1([&](int q) { return a.dstq[q] + i; }, d, uint32_t(i), seed.get());
    if (CHECK)
      check_node(sums, o.rho, o.ux, o.uy, o.uz, a.C.rho0, static_cast<float*>(a.cb.uprev) + i,
                 int64_t(a.plane) * a.nz);
  }
  if (CHECK) block_sums(sums, check_row(a.cb), a.cb.flag);
}

}  // namespace

// Lattices with the unit rates omega_9..18 take the pair kernel where it is
// the faster one (pair_pays), the others one node per thread.
cudaError_t launch_step_f16sr(const void* src, void* dst, const Geom& g, const PhysParams& P,
                              const CheckBufs& cb, bool check, dim3 block, int64_t step,
                              const unsigned* base, cudaStream_t st) {
  const StepArgs<__half, float> a = step_args<__half, float>(src, dst, g, P, cb);
  const StepSeed seed{unsigned(uint64_t(step)), base};
  const bool unit = unit_rates(P);
  if (unit && pair_pays(g, false))
    return launch_step_pair<PAIR_SR>(a, PairExtra{nullptr, nullptr, seed}, P.has_force != 0,
                                     check, block, st);
  const dim3 grid((g.nx + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y, g.nz);
  void (*kernel)(const StepArgs<__half, float>, const StepSeed) = nullptr;
#define CLBM_SR(F, C_) kernel = unit ? step_sr_kernel<F, C_, true> : step_sr_kernel<F, C_, false>
  if (P.has_force) {
    if (check) CLBM_SR(true, true);
    else CLBM_SR(true, false);
  } else {
    if (check) CLBM_SR(false, true);
    else CLBM_SR(false, false);
  }
#undef CLBM_SR
  return pdl_launch(kernel, grid, block, st, a, seed);
}

}  // namespace clbm
