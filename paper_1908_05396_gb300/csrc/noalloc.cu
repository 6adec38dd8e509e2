// noalloc.cu -- one check step between caller-owned buffers, allocating nothing.
//
// Some callers cannot allocate device memory when they step: a solver embedded
// in a host application that owns a fixed device-memory pool handed out at
// start-up, code running where cudaMalloc is forbidden (inside a memory-budget
// manager, or a framework that has already reserved all of the device), or
// callers that must never stall on the allocator's implicit synchronisation.
// clbm_step_noalloc() serves them: it runs the same fused step as a check step
// of clbm_step() on buffers the caller passes in, and keeps the per-block
// partial sums of its FP64 reductions in a fixed file-scope device array
// instead of memory obtained from cudaMalloc.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>

#include "../../include/clbm.h"
#include "kernels.cuh"
#include "validate.h"

namespace clbm {
namespace {

// Partial sums of one call: 4 doubles per thread block of the step.  Every
// GPU that loads the library holds this array (2 MiB) until the process ends.
constexpr int NOALLOC_MAX_BLOCKS = 65536;
static __device__ __align__(256) double g_noalloc_partials[NOALLOC_MAX_BLOCKS * 4];

constexpr int MAX_DEVICES = 64;
std::mutex g_mu;
double* g_partials_ptr[MAX_DEVICES] = {};

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device with that device current.
cudaError_t scratch_address(int dev, double** out) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  if (!g_partials_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
    if (e != cudaSuccess) return e;
    g_partials_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_partials_ptr[dev];
  return cudaSuccess;
}

// The check step of step_kernel, with each block writing its partial sums
// (sum|u - uprev|^2, sum|u|^2, sum(rho - rho0), divergence) to its own slot of
// the scratch array instead of adding them atomically.
template <typename S, typename R, bool FORCE>
__global__ void __launch_bounds__(256) step_partials_kernel(const StepArgs<S, R> a,
                                                            double* partials) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  CheckSums sums;
  if (x < a.nx && y < a.ny) {
    const int i = z * a.plane + y * a.pitch + x;
    R d[Q];
    pull_node(a, x, y, z, i, d);
    NodeOut<R> o;
    collide<R, FORCE, pair_out<S>(), log2_scale<S>(), true>(a.C, d, o);
#pragma unroll
    for (int q = 0; q < Q; ++q) a.dstq[q][i] = Codec<S, R>::enc(d[q], R(1));
    check_node(sums, o.rho, o.ux, o.uy, o.uz, a.C.rho0, static_cast<R*>(a.cb.uprev) + i,
               int64_t(a.plane) * a.nz);
  }
  // Fixed-order block reduction, so that the result does not depend on
  // scheduling.
  __shared__ double sm[8][3];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = int(blockDim.x * blockDim.y) >> 5;
  const double v = warp_sums(sums);
  if (lane == 0) sm[warp][0] = v;
  if (lane == 16) sm[warp][1] = v;
  if (lane == 8) sm[warp][2] = v;
  const int bad = __syncthreads_or(sums.bad);
  if (tid < 4) {
    double t = tid < 3 ? sm[0][tid < 3 ? tid : 0] : double(bad != 0);
    for (int w = 1; w < nwarp && tid < 3; ++w) t += sm[w][tid];
    const int64_t b = (int64_t(blockIdx.z) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    partials[b * 4 + tid] = t;
  }
}

// Second pass: one block sums the nblocks partials in a fixed order and
// writes the four results (the divergence entry as 0 or 1).  Thread t takes
// entry t & 3 of every 256th block's partials, so that a warp reads whole
// lines; four sums a thread keep its loads in flight.
constexpr int FINISH_THREADS = 1024;
__global__ void __launch_bounds__(FINISH_THREADS) finish_kernel(
    const double* __restrict__ partials, int nblocks, double* stats) {
  __shared__ double sm[FINISH_THREADS];
  const int t = int(threadIdx.x), n = 4 * nblocks;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (int b = t; b < n; b += 4 * FINISH_THREADS)
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (b + k * FINISH_THREADS < n) a[k] += partials[b + k * FINISH_THREADS];
  sm[t] = (a[0] + a[1]) + (a[2] + a[3]);
  __syncthreads();
  for (int s = FINISH_THREADS / 2; s >= 4; s >>= 1) {
    if (t < s) sm[t] += sm[t + s];
    __syncthreads();
  }
  if (t < 4) stats[t] = t < 3 ? sm[t] : (sm[t] > 0.0 ? 1.0 : 0.0);
}

template <typename S, typename R>
cudaError_t launch_noalloc(const void* src, void* dst, const Geom& g, const PhysParams& P,
                           void* uprev, double* partials, double* stats, dim3 grid, dim3 block,
                           cudaStream_t st) {
  CheckBufs cb{};
  cb.uprev = uprev;
  // (dense rows; the entry point takes the unit rates omega_9..18 only)
  StepArgs<S, R> a = step_args<S, R>(src, dst, g, P, cb);
  if (P.has_force) step_partials_kernel<S, R, true><<<grid, block, 0, st>>>(a, partials);
  else step_partials_kernel<S, R, false><<<grid, block, 0, st>>>(a, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  finish_kernel<<<1, FINISH_THREADS, 0, st>>>(partials, int(grid.x * grid.y * grid.z), stats);
  return cudaGetLastError();
}

int noalloc_fail(int code, const char* msg) {
  set_unbound_error(msg);
  return code;
}

}  // namespace
}  // namespace clbm

using namespace clbm;

extern "C" int clbm_step_noalloc(const clbm_domain* d, double K, double n, const double U_lid[3],
                                 const double body_force[3], clbm_dtype dtype, const void* src,
                                 void* dst, void* u_prev, double* stats) {
  if (!d || !src || !dst || !u_prev || !stats)
    return noalloc_fail(CLBM_ERR_ARG, "null domain or buffer");
  if (src == dst) return noalloc_fail(CLBM_ERR_ARG, "src and dst must be different buffers");
  if (dtype == CLBM_F16R)
    return noalloc_fail(CLBM_ERR_UNSUPPORTED, "the F16R form is not available here");
  if (dtype != CLBM_F64 && dtype != CLBM_F32 && dtype != CLBM_F16S)
    return noalloc_fail(CLBM_ERR_ARG, "unknown dtype");
  std::string why;
  double U[3];
  if (!check_domain(d, U_lid, U, why)) return noalloc_fail(CLBM_ERR_ARG, why.c_str());
  double rho0, nu_min, nu_max;
  domain_defaults(d, &rho0, &nu_min, &nu_max);
  if (!check_phys(K, n, nu_min, nu_max, why)) return noalloc_fail(CLBM_ERR_ARG, why.c_str());
  if (!check_force(body_force, why)) return noalloc_fail(CLBM_ERR_ARG, why.c_str());

  // Dense layout: pop[q][z][y][x] with no padding, u_prev[3][z][y][x].
  Geom g{};
  g.nx = d->nx;
  g.ny = d->ny;
  g.nz = d->nz;
  g.pitch = d->nx;
  g.plane = int64_t(d->nx) * d->ny;
  g.qstride = g.plane * d->nz;
  g.facebits = 0;
  for (int f = 0; f < 6; ++f) g.facebits |= unsigned(d->face[f]) << (2 * f);
  for (int a = 0; a < 3; ++a) g.U[a] = U[a];
  g.rho0 = rho0;
  PhysParams P{};
  fill_params(P, K, n, body_force, rho0, nu_min, nu_max, dtype);
  const dim3 block(32, 4, 1);
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  const int64_t nblocks = int64_t(grid.x) * grid.y * grid.z;
  if (nblocks > NOALLOC_MAX_BLOCKS) {
    char msg[256];
    snprintf(msg, sizeof(msg),
             "lattice needs %lld thread blocks of 32x4 nodes; the fixed scratch of "
             "clbm_step_noalloc holds partial sums for at most %d (about 8.4 million nodes)",
             (long long)nblocks, NOALLOC_MAX_BLOCKS);
    return noalloc_fail(CLBM_ERR_ARG, msg);
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  double* partials = nullptr;
  cudaStream_t st = static_cast<cudaStream_t>(d->stream);
  if (e == cudaSuccess) e = scratch_address(dev, &partials);
  if (e != cudaSuccess) {
    // The first call on a device looks the scratch address up, which a
    // stream capture in progress does not allow.
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
      std::string m = std::string(cudaGetErrorString(e)) +
                      ": the first clbm_step_noalloc call on a device must come before any "
                      "stream capture";
      return noalloc_fail(CLBM_ERR_CUDA, m.c_str());
    }
    return noalloc_fail(CLBM_ERR_CUDA, cudaGetErrorString(e));
  }
  switch (dtype) {
    case CLBM_F64:
      e = launch_noalloc<double, double>(src, dst, g, P, u_prev, partials, stats, grid, block, st);
      break;
    case CLBM_F32:
      e = launch_noalloc<float, float>(src, dst, g, P, u_prev, partials, stats, grid, block, st);
      break;
    default:
      e = launch_noalloc<__half, float>(src, dst, g, P, u_prev, partials, stats, grid, block, st);
      break;
  }
  if (e != cudaSuccess) return noalloc_fail(CLBM_ERR_CUDA, cudaGetErrorString(e));
  return CLBM_OK;
}
