// kernels.cuh -- fused pull-stream + cascaded-collision step and its helpers.
//
// Storage: structure of arrays pop[q][z][y][x] with a padded row pitch, two
// buffers (A-B).  A thread owns one node: it pulls the 19 post-collision
// populations of its upwind neighbours from buffer A (Eq. cascadedstreaming1),
// resolving walls, the lid and periodic faces from its own index, collides
// (Sec. 3) and writes the 19 results to its own slot of buffer B.  Every
// read and write of a warp covers consecutive x, so the accesses coalesce;
// the +/-x directions are offset by one element, which costs one extra
// sector per warp in L1/L2 but no extra DRAM traffic.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "collide.cuh"
#include "launch.h"

namespace clbm {

// ---- storage codecs: stored value <-> deviation f - w rho0 -----------------
template <typename S, typename R> struct Codec;
template <typename R> struct Codec<double, R> {
  static __device__ __forceinline__ R dec(double v, R) { return R(v); }
  static __device__ __forceinline__ double enc(R v, R) { return double(v); }
};
template <typename R> struct Codec<float, R> {
  static __device__ __forceinline__ R dec(float v, R) { return R(v); }
  static __device__ __forceinline__ float enc(R v, R) { return float(v); }
};
template <typename R> struct Codec<__half, R> {
  // (f - w rho0) * 1024 in FP16, round to nearest even.  The power-of-two
  // scale is exact and lifts deviations down to ~6e-8 out of the FP16
  // subnormal range while keeping |f - w rho0| < 64 representable.  The
  // kernels work on the scaled deviations directly (log2_scale): the scale
  // is folded into the collision's constants, so decoding and encoding are
  // plain conversions.
  static __device__ __forceinline__ R dec(__half v, R) { return R(__half2float(v)); }
  static __device__ __forceinline__ __half enc(R v, R) { return __float2half_rn(float(v)); }
};

// log2 of the factor by which storage type S holds the deviations f - w rho0
// (and by which the kernels carry them): 10 for FP16, 0 otherwise.
template <typename S>
__host__ __device__ constexpr int log2_scale() {
  return std::is_same<S, __half>::value ? 10 : 0;
}

// Whether the collision rebuilds the populations of storage type S from its
// pair values (see collide): for FP16 storage, whose decoded values sum
// without rounding, and for FP64, whose rounding stays far below every
// tolerance; FP32 storage takes one added correction per population.
template <typename S>
__host__ __device__ constexpr bool pair_out() {
  return std::is_same<S, __half>::value || std::is_same<S, double>::value;
}

// Collision constants for deviations carried scaled by lam (a power of two;
// see collide_rates): the rest density and the force of the scaled moments, and
// 3K and its logarithm so that nu and the omega solve come out unscaled.
template <typename R>
inline CollideConst<R> make_const(const PhysParams& P, double lam = 1.0) {
  const double L2E = 1.4426950408889634074;
  CollideConst<R> C;
  C.rho0 = R(P.rho0);
  C.rhoS = R(lam * P.rho0);
  C.r30 = R(lam * P.rho0 / 3.0);
  for (int a = 0; a < 3; ++a) C.FS[a] = R(lam * P.F[a]);
  C.K3 = R(3.0 * P.K * lam);
  C.nu_min = R(P.nu_min);
  C.nu_max = R(P.nu_max);
  const double clog = P.logK3 + log(lam) + 0.5 * (P.n - 1.0) * log(9.0);
  if constexpr (std::is_same<R, double>::value) {
    C.clog = clog;
    C.eh = 0.5 * (P.n - 1.0);
    C.nm1 = P.n - 1.0;
    C.tlo = 3.0 * P.nu_min;
    C.thi = 3.0 * P.nu_max;
  }
  C.n = float(P.n);
  C.rn = float(1.0 / P.n);
  C.ehalf = float(0.5 * (P.n - 1.0));
  C.clog2 = float(clog * L2E);
  C.ylo2 = float(P.ylo * L2E);
  C.yhi2 = float(P.yhi * L2E);
  // the invariant carries lam^2: the same shear rate for every scale
  C.g2lo = float(1e-36 * lam * lam);
  C.newtonian = P.newtonian;
  C.has_force = P.has_force;
  const double* w = P.omega_high;  // omega_9 .. omega_18
  C.c9 = R(-w[0] / 126.0);
  C.c10 = R(0.125 * w[1]);
  C.c11 = R(0.125 * w[2]);
  C.c12 = R(0.125 * w[3]);
  C.c13 = R(0.125 * w[4]);
  C.c14 = R(0.125 * w[5]);
  C.c15 = R(0.125 * w[6]);
  C.c16 = R(w[7] / 12.0);
  C.c17 = R(w[8] / 24.0);
  C.c18 = R(0.125 * w[9]);
  C.cB = R(w[0] * w[0] / 6.0);
  return C;
}

// ---- check-step sums ----------------------------------------------------------
// FP64 instructions run at 1/64 of the FP32 rate, so a check step spends as few
// as it can: conversions are integer operations (to64), the finiteness test is
// made in the math type, and a warp's three sums share their reduction steps.
// The blocks' sums go to CheckBufs::rows rows, so that no address takes more
// than a few hundred atomic additions.  With one row, a tree per sum and the
// hardware's conversions a check step of 128^3 took 247 us in FP32, 211 in F16S
// and 162 in F16R, against 100, 76 and 88 now (a plain step: 47, 31 and 56).

// A node's part of the sums over the lattice, in FP64: sum|u - u_prev|^2,
// sum|u|^2, sum(rho - rho0), and whether the node diverged.
struct CheckSums {
  double du2 = 0.0, uu = 0.0, dr = 0.0;
  int bad = 0;
};

// Adds a node with the results (rho, u); up points at the node's x velocity of
// the previous check (components nst apart), which is replaced.
template <typename R>
__device__ __forceinline__ void check_node(CheckSums& s, R rho, R ux, R uy, R uz, R rho0, R* up,
                                           int64_t nst) {
  const R px = up[0], py = up[nst], pz = up[2 * nst];
  up[0] = ux;
  up[nst] = uy;
  up[2 * nst] = uz;
  const double x = to64(ux), y = to64(uy), z = to64(uz);
  const double ex = x - to64(px), ey = y - to64(py), ez = z - to64(pz);
  s.du2 = fma(ex, ex, fma(ey, ey, fma(ez, ez, s.du2)));
  s.uu = fma(x, x, fma(y, y, fma(z, z, s.uu)));
  s.dr += to64(rho) - to64(rho0);
  s.bad |= !(rho > R(0.5) && rho < R(2.0)) || !(fabs(ux) < R(1e30)) || !(fabs(uy) < R(1e30)) ||
           !(fabs(uz) < R(1e30));
}

// The warp's three sums: du2 in lane 0, uu in lane 16, dr in lane 8.  The
// first two exchanges each fold two quantities into the halves of the warp.
__device__ __forceinline__ double warp_sums(const CheckSums& s) {
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = int(threadIdx.x + threadIdx.y * blockDim.x) & 31;
  const bool h = lane & 16, o = lane & 8;
  const double a = (h ? s.uu : s.du2) + __shfl_xor_sync(ALL, h ? s.du2 : s.uu, 16);
  const double b = s.dr + __shfl_xor_sync(ALL, s.dr, 16);
  double c = (o ? b : a) + __shfl_xor_sync(ALL, o ? a : b, 8);
#pragma unroll
  for (int k = 4; k > 0; k >>= 1) c += __shfl_xor_sync(ALL, c, k);
  return c;
}

// Adds the block's sums to a row of acc (4 doubles a row: the three sums) and
// raises the flag if a node diverged.  Called by every thread of the block.
__device__ __forceinline__ void block_sums(const CheckSums& s, double* row, int* flag) {
  __shared__ double sm[8][3];
  const int t = int(threadIdx.x + threadIdx.y * blockDim.x), lane = t & 31, warp = t >> 5;
  const double v = warp_sums(s);
  if (lane == 0) sm[warp][0] = v;
  if (lane == 16) sm[warp][1] = v;
  if (lane == 8) sm[warp][2] = v;
  const int bad = __syncthreads_or(s.bad);
  if (t < 3) {
    double a = sm[0][t];
    for (int w = 1; w < int(blockDim.x * blockDim.y) >> 5; ++w) a += sm[w][t];
    atomicAdd(row + t, a);
  }
  if (t == 0 && bad) atomicOr(flag, 1);
  __syncthreads();
}
// The row of a block of a lone lattice's check step.
__device__ __forceinline__ double* check_row(const CheckBufs& cb) {
  const unsigned blk = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  return cb.acc + 4 * (blk & unsigned(cb.rows - 1));
}

// ---- the fused step ---------------------------------------------------------
// Everything one step launch needs, precomputed on the host in the math
// precision R (no double arithmetic is left in the FP32 kernels).
template <typename S, typename R>
struct StepArgs {
  const S* srcq[Q];  // srcq[q][i]: stored f~_q of the upwind neighbour of node i
  S* dstq[Q];        // dstq[q][i]: slot of direction q of node i
  const S* src;      // source buffer base (bounce-back and general path)
  int64_t qstride;
  int nx, ny, nz, pitch, plane;
  unsigned facebits;
  int zrev;          // 1: planes in descending z (every other step, see launch_step_t)
  R lidc[Q];         // 6 w_q rho0 (e_q . U_lid): lid momentum correction
  CollideConst<R> C;
  CheckBufs cb;
};

// The faces a node lies on.  Bits 0..5 stand for the faces -x, +x, -y, +y,
// -z, +z: `wall` has those of the node's faces that are walls or lids, `lid`
// the lids among them; wrap[k] is the index offset that brings a step across
// face k back into the lattice when the node lies on that face (else 0).
struct Faces {
  unsigned wall, lid;
  int wrap[6];
};
__device__ __forceinline__ Faces faces_of(int x, int y, int z, int nx, int ny, int nz, int pitch,
                                          int plane, unsigned fb) {
  const bool at[6] = {x == 0, x == nx - 1, y == 0, y == ny - 1, z == 0, z == nz - 1};
  const int len[3] = {nx, ny * pitch, nz * plane};
  Faces f;
  f.wall = f.lid = 0u;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const unsigned kind = (fb >> (2 * k)) & 3u;
    if (at[k] && kind != BC_PERIODIC) f.wall |= 1u << k;
    if (at[k] && kind == BC_LID) f.lid |= 1u << k;
    f.wrap[k] = at[k] ? (k & 1 ? -len[k / 2] : len[k / 2]) : 0;
  }
  return f;
}
// Faces that a step along -e_q (the upwind side) can cross; the downwind side
// of q is the upwind side of opp(q).
__host__ __device__ constexpr unsigned up_faces(int q) {
  return (cx(q) == 1 ? 1u : cx(q) == -1 ? 2u : 0u) | (cy(q) == 1 ? 4u : cy(q) == -1 ? 8u : 0u) |
         (cz(q) == 1 ? 16u : cz(q) == -1 ? 32u : 0u);
}
// Index offset of the periodic wrap of a step along -e_q.
__device__ __forceinline__ int up_wrap(const Faces& f, int q) {
  int w = 0;
  if (cx(q)) w += f.wrap[cx(q) == 1 ? 0 : 1];
  if (cy(q)) w += f.wrap[cy(q) == 1 ? 2 : 3];
  if (cz(q)) w += f.wrap[cz(q) == 1 ? 4 : 5];
  return w;
}

// Pull of all 19 directions into node (x, y, z) with index i, for a node on
// any face: the upwind node's value, across a periodic face the wrapped
// node's, or, where any crossed face is a wall or the lid, halfway bounce-back
// from the node's own opposite population, plus the lid term when a crossed
// face is the lid.  The rule selects an address, so the 19 loads are issued
// together; branching to a load per rule exposed their latency one after the
// other, in a small lattice most of the step (32^3 F16S 8.3 us a step, 4.6
// with the addresses selected, FP32 6.1 and 4.3) and in a large one the tail
// that the face blocks formed (128^3 F16S 38.6 and 30.7, F16R 61 and 55, FP32
// 53 and 50).
template <typename S, typename R>
__device__ __forceinline__ void pull_face(const S* __restrict__ src, int64_t qstride, int nx,
                                          int ny, int nz, int pitch, int plane, unsigned fb,
                                          int x, int y, int z, int i, const R* lidc, R (&d)[Q]) {
  const Faces f = faces_of(x, y, z, nx, ny, nz, pitch, plane, fb);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const bool bounce = (f.wall & up_faces(q)) != 0;
    const int j = i - (cz(q) * plane + cy(q) * pitch + cx(q)) + up_wrap(f, q);
    const S* p = src + (bounce ? int64_t(opp(q)) * qstride : int64_t(q) * qstride);
    d[q] = Codec<S, R>::dec(p[bounce ? i : j], R(1));
    if (f.lid & up_faces(q)) d[q] += lidc[q];
  }
}

// Pull of node (x, y, z) with index i of a two-buffer lattice: a warp off
// every face loads its 19 upwind values directly, any other goes through
// pull_face as a whole (patching the lanes on an x face after direct loads
// costs a second, dependent round of loads: 32^3 FP32 4.3 us a step against
// 2.6, 128^3 50.4 against 48.4).
template <typename S, typename R>
__device__ __forceinline__ void pull_node(const StepArgs<S, R>& a, int x, int y, int z, int i,
                                          R (&d)[Q]) {
  const bool inner = y > 0 && y < a.ny - 1 && z > 0 && z < a.nz - 1 && x > 0 && x < a.nx - 1;
  if (__all_sync(__activemask(), inner)) {
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = Codec<S, R>::dec(a.srcq[q][i], R(1));
  } else {
    pull_face<S, R>(a.src, a.qstride, a.nx, a.ny, a.nz, a.pitch, a.plane, a.facebits, x, y, z, i,
                    a.lidc, d);
  }
}

// Programmatic dependent launch between consecutive steps.  A step launched
// with the programmatic stream-serialisation attribute may be scheduled
// while the previous step's last blocks still run: each of its threads waits
// here until the previous grid has completed and its writes are visible,
// before any global access, and then allows the next step to be scheduled.
// The next grid is only scheduled once every block of this one has passed
// this point (or exited), so its waiting blocks never take SM slots that a
// block of this grid still needs.  Without the attribute both are no-ops.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// Launch a kernel whose threads start with pdl_enter(), with the programmatic
// stream-serialisation attribute (compiled out with -DCLBM_NO_PDL) and
// `smem` bytes of dynamic shared memory.
template <typename... KArgs, typename... Args>
inline cudaError_t pdl_launch_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                   cudaStream_t st, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
#ifdef CLBM_NO_PDL
  cfg.numAttrs = 0;
#else
  cfg.numAttrs = 1;
#endif
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}
template <typename... KArgs, typename... Args>
inline cudaError_t pdl_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st,
                              const Args&... args) {
  return pdl_launch_smem(kernel, grid, block, 0, st, args...);
}

// One time step.  CHECK = true also writes u into uprev (after reading
// the previous check's value there) and reduces sum|u - uprev|^2, sum|u|^2,
// sum(rho - rho0) and a divergence flag in FP64.
// CAP = true caps registers so that four 256-thread (or eight 128-thread)
// blocks fit on an SM: more warps to hide DRAM latency, at the risk of
// spills; the autotuner decides.
// UNIT: relaxation rates omega_9..18 all 1 (collide_unit); lattices with other
// rates have no register-capped variant.
template <typename S, typename R, bool FORCE, bool CHECK, bool CAP, bool UNIT>
__global__ void __launch_bounds__(256, CAP ? 4 : 1) step_kernel(const StepArgs<S, R> a) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = a.zrev ? a.nz - 1 - int(blockIdx.z) : int(blockIdx.z);
  const bool active = x < a.nx && y < a.ny;
  if (!CHECK && !active) return;
  CheckSums sums;
  if (active) {
    const int i = z * a.plane + y * a.pitch + x;
    R d[Q];
    pull_node(a, x, y, z, i, d);
    NodeOut<R> o;
    collide<R, FORCE, pair_out<S>(), log2_scale<S>(), UNIT>(a.C, d, o);
#pragma unroll
    for (int q = 0; q < Q; ++q) a.dstq[q][i] = Codec<S, R>::enc(d[q], R(1));
    if (CHECK)
      check_node(sums, o.rho, o.ux, o.uy, o.uz, a.C.rho0, static_cast<R*>(a.cb.uprev) + i,
                 int64_t(a.plane) * a.nz);
  }
  if (CHECK) block_sums(sums, check_row(a.cb), a.cb.flag);
}

// Output arrays of the macroscopic fields, unpadded [z][y][x]; any may be null.
struct FieldsOut {
  double *rho, *u, *gd;
};
template <typename R>
__device__ __forceinline__ void write_fields(const FieldsOut& f, const NodeOut<R>& o, int nx,
                                             int ny, int nz, int x, int y, int z) {
  const int64_t N = int64_t(nx) * ny * nz;
  const int64_t k = (int64_t(z) * ny + y) * nx + x;
  if (f.rho) f.rho[k] = to64(o.rho);
  if (f.u) {
    f.u[k] = to64(o.ux);
    f.u[N + k] = to64(o.uy);
    f.u[2 * N + k] = to64(o.uz);
  }
  if (f.gd) f.gd[k] = to64(o.gamma_dot);
}

// Macroscopic fields of the current state (pull + moments + omega solve, the
// last only for |gamma_dot|).
template <typename S, typename R, bool FORCE>
__global__ void __launch_bounds__(256) fields_kernel(const StepArgs<S, R> a, const FieldsOut f) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= a.nx || y >= a.ny) return;
  R d[Q];
  pull_node(a, x, y, z, z * a.plane + y * a.pitch + x, d);
  NodeOut<R> o;
  node_fields<R, FORCE, log2_scale<S>()>(a.C, d, f.gd != nullptr, o);
  write_fields(f, o, a.nx, a.ny, a.nz, x, y, z);
}

// Collide M independent nodes given as plain FP64 populations [q][node].
template <typename S, typename R, bool FORCE>
__global__ void collide_nodes_kernel(CollideConst<R> C, double rho0, const double* __restrict__ fin,
                                     double* __restrict__ fout, double* rho,
                                     double* u, double* gd, int64_t M) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= M) return;
  const double lam = double(1 << log2_scale<S>());
  R d[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const R dev = R((fin[q * M + k] - wt<double>(q) * rho0) * lam);
    d[q] = Codec<S, R>::dec(Codec<S, R>::enc(dev, R(lam)), R(lam));
  }
  NodeOut<R> o;
  collide<R, FORCE, pair_out<S>(), log2_scale<S>(), true>(C, d, o);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const R st = Codec<S, R>::dec(Codec<S, R>::enc(d[q], R(lam)), R(lam));
    fout[q * M + k] = double(st) / lam + wt<double>(q) * rho0;
  }
  if (rho) rho[k] = double(o.rho);
  if (u) {
    u[k] = double(o.ux);
    u[M + k] = double(o.uy);
    u[2 * M + k] = double(o.uz);
  }
  if (gd) gd[k] = double(o.gamma_dot);
}

// The local relaxation rate omega_nu and |gamma_dot| of M nodes from their
// density and non-equilibrium moments m^(1)_4..9 ([6][node], FP64), solved
// in the math precision R exactly as the collision does.
template <typename R>
__global__ void omega_nodes_kernel(CollideConst<R> C, const double* __restrict__ rho_in,
                                   const double* __restrict__ m, double* omega, double* gd,
                                   int64_t M) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= M) return;
  const R rho = R(rho_in[k]);
  const R rinv = rrcp<R>(rho);
  R A, B;
  strain_AB(C, R(m[k]), R(m[M + k]), R(m[2 * M + k]), R(m[3 * M + k]), R(m[4 * M + k]),
            R(m[5 * M + k]), A, B);
  const R w = omega_nu(C, rho, rinv, A, B);
  omega[k] = double(w);
  if (gd) gd[k] = double(shear_rate(rinv, w, A, B));
}

// Stored populations <-> plain FP64 f in the unpadded layout [q][z][y][x]: one
// thread per node, all directions (one per population spent four 64-bit
// divisions on its place, and the import a fifth on the scale, a power of two).
template <typename S>
__global__ void __launch_bounds__(128) export_kernel(const S* __restrict__ src, Geom g,
                                                     double rho0, double inv_scale,
                                                     double* __restrict__ out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  const int64_t N = int64_t(g.nx) * g.ny * g.nz, k = (int64_t(z) * g.ny + y) * g.nx + x;
  const int64_t i = int64_t(z) * g.plane + int64_t(y) * g.pitch + x;
#pragma unroll
  for (int q = 0; q < Q; ++q)
    out[q * N + k] = double(Codec<S, double>::dec(src[q * g.qstride + i], inv_scale)) * inv_scale +
                     wt<double>(q) * rho0;
}

template <typename S>
__global__ void __launch_bounds__(128) import_kernel(const double* __restrict__ in, Geom g,
                                                     double rho0, double scale,
                                                     S* __restrict__ dst) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  const int64_t N = int64_t(g.nx) * g.ny * g.nz, k = (int64_t(z) * g.ny + y) * g.nx + x;
  const int64_t i = int64_t(z) * g.plane + int64_t(y) * g.pitch + x;
#pragma unroll
  for (int q = 0; q < Q; ++q)
    dst[q * g.qstride + i] =
        Codec<S, double>::enc((in[q * N + k] - wt<double>(q) * rho0) * scale, scale);
}

// The arguments of a two-buffer step from src to dst.
template <typename S, typename R>
StepArgs<S, R> step_args(const void* src, void* dst, const Geom& g, const PhysParams& P,
                         const CheckBufs& cb) {
  StepArgs<S, R> a;
  const S* s = static_cast<const S*>(src);
  S* d = static_cast<S*>(dst);
  const double lam = double(1 << log2_scale<S>());
  for (int q = 0; q < Q; ++q) {
    const int64_t off = int64_t(cz(q)) * g.plane + int64_t(cy(q)) * g.pitch + cx(q);
    // address arithmetic through integers: the shifted base may precede the
    // buffer, only base + i of a node in the box is dereferenced
    a.srcq[q] = reinterpret_cast<const S*>(reinterpret_cast<uintptr_t>(s) +
                                            (int64_t(q) * g.qstride - off) * int64_t(sizeof(S)));
    a.dstq[q] = d + int64_t(q) * g.qstride;
    a.lidc[q] = R(6.0 * wt<double>(q) * g.rho0 * lam *
                  (cx(q) * g.U[0] + cy(q) * g.U[1] + cz(q) * g.U[2]));
  }
  a.src = s;
  a.qstride = g.qstride;
  a.nx = g.nx;
  a.ny = g.ny;
  a.nz = g.nz;
  a.pitch = g.pitch;
  a.plane = int(g.plane);
  a.facebits = g.facebits;
  // Blocks run roughly in launch order, z planes last, so a step ends with
  // its highest planes still in L2.  Sweeping z downward on every other step
  // (the steps that write the lower-addressed of the two buffers) makes the
  // next step read those planes first, from L2.
  a.zrev = reinterpret_cast<uintptr_t>(dst) < reinterpret_cast<uintptr_t>(src) ? 1 : 0;
  a.C = make_const<R>(P, lam);
  a.cb = cb;
  return a;
}

}  // namespace clbm

#include "tma_step.cuh"
#include "inplace.cuh"
#include "pair.cuh"

namespace clbm {

// ---- host-side launchers, instantiated once per storage type --------------

template <typename S, typename R>
cudaError_t launch_step_t(const void* src, void* dst, const Geom& g, const PhysParams& P,
                          const CheckBufs& cb, bool check, dim3 block, int npt,
                          cudaStream_t st) {
  StepArgs<S, R> a = step_args<S, R>(src, dst, g, P, cb);
  // npt: 1 or 2 nodes per thread; +4 selects the register-capped variant;
  // TMA_NPT + 32 v the TMA-staged kernel of shape v (check steps take the
  // plain kernel with the same block).
  if constexpr (std::is_same<R, float>::value && !std::is_same<S, double>::value) {
    if ((npt & TMA_NPT) && !check && unit_rates(P))
      return launch_step_tma<S>(a, src, g, P.has_force != 0, npt >> 5, cb.flag + 1, st);
  }
  const bool cap = (npt & 4) != 0;
  npt &= 3;
  const dim3 grid((g.nx + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y, g.nz);
  const int fc = (P.has_force ? 2 : 0) + (check ? 1 : 0);
  void (*kernel)(const StepArgs<S, R>) = nullptr;
  if (!unit_rates(P)) {
    kernel = fc == 3   ? step_kernel<S, R, true, true, false, false>
             : fc == 2 ? step_kernel<S, R, true, false, false, false>
             : fc == 1 ? step_kernel<S, R, false, true, false, false>
                       : step_kernel<S, R, false, false, false, false>;
    return pdl_launch(kernel, grid, block, st, a);
  }
  if constexpr (std::is_same<S, __half>::value) {
    if (npt == 2 || pair_pays(g, false))
      return launch_step_pair<PAIR_RN>(a, PairExtra{}, P.has_force != 0, check, block, st);
    kernel = fc == 3   ? step_kernel<S, R, true, true, true, true>
             : fc == 2 ? step_kernel<S, R, true, false, true, true>
             : fc == 1 ? step_kernel<S, R, false, true, true, true>
                       : step_kernel<S, R, false, false, true, true>;
    return pdl_launch(kernel, grid, block, st, a);
  } else {
    if (cap)
      kernel = fc == 3   ? step_kernel<S, R, true, true, true, true>
               : fc == 2 ? step_kernel<S, R, true, false, true, true>
               : fc == 1 ? step_kernel<S, R, false, true, true, true>
                         : step_kernel<S, R, false, false, true, true>;
    else
      kernel = fc == 3   ? step_kernel<S, R, true, true, false, true>
               : fc == 2 ? step_kernel<S, R, true, false, false, true>
               : fc == 1 ? step_kernel<S, R, false, true, false, true>
                         : step_kernel<S, R, false, false, false, true>;
    return pdl_launch(kernel, grid, block, st, a);
  }
}

template <typename S, typename R>
cudaError_t launch_fields_t(const void* src, const Geom& g, const PhysParams& P, double* rho,
                            double* u, double* gd, cudaStream_t st) {
  const dim3 block(32, 4);
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  const StepArgs<S, R> a = step_args<S, R>(src, nullptr, g, P, CheckBufs{});
  const FieldsOut f{rho, u, gd};
  if (P.has_force) fields_kernel<S, R, true><<<grid, block, 0, st>>>(a, f);
  else fields_kernel<S, R, false><<<grid, block, 0, st>>>(a, f);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_collide_nodes_t(const PhysParams& P, const double* fin, double* fout,
                                   double* rho, double* u, double* gd, int64_t M,
                                   cudaStream_t st) {
  const int b = 128;
  const unsigned grid = unsigned((M + b - 1) / b);
  const CollideConst<R> C = make_const<R>(P, double(1 << log2_scale<S>()));
  if (P.has_force)
    collide_nodes_kernel<S, R, true><<<grid, b, 0, st>>>(C, P.rho0, fin, fout, rho, u, gd, M);
  else
    collide_nodes_kernel<S, R, false><<<grid, b, 0, st>>>(C, P.rho0, fin, fout, rho, u, gd, M);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_omega_nodes_t(const PhysParams& P, const double* rho, const double* m,
                                 double* omega, double* gd, int64_t M, cudaStream_t st) {
  const int b = 128;
  omega_nodes_kernel<R><<<unsigned((M + b - 1) / b), b, 0, st>>>(make_const<R>(P), rho, m, omega, gd, M);
  return cudaGetLastError();
}

inline dim3 node_grid(const Geom& g) {
  return dim3((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
}

template <typename S>
cudaError_t launch_export_t(const void* src, const Geom& g, double rho0, double inv_scale,
                            double* out, cudaStream_t st) {
  export_kernel<S><<<node_grid(g), dim3(32, 4), 0, st>>>(static_cast<const S*>(src), g, rho0,
                                                         inv_scale, out);
  return cudaGetLastError();
}

template <typename S>
cudaError_t launch_import_t(const double* in, const Geom& g, double rho0, double inv_scale,
                            void* dst, cudaStream_t st) {
  import_kernel<S><<<node_grid(g), dim3(32, 4), 0, st>>>(in, g, rho0, 1.0 / inv_scale,
                                                         static_cast<S*>(dst));
  return cudaGetLastError();
}

}  // namespace clbm

// Defines the launchers of launch.h for one storage type S with math type R.
#define CLBM_DEFINE_LAUNCHERS(SUFFIX, S, R)                                                   \
  namespace clbm {                                                                            \
  cudaError_t launch_step_##SUFFIX(const void* src, void* dst, const Geom& g,                 \
                                   const PhysParams& P, const CheckBufs& cb, bool check,      \
                                   dim3 block, int npt, cudaStream_t st) {                    \
    return launch_step_t<S, R>(src, dst, g, P, cb, check, block, npt, st);                    \
  }                                                                                           \
  cudaError_t launch_fields_##SUFFIX(const void* src, const Geom& g, const PhysParams& P,     \
                                     double* rho, double* u, double* gd, cudaStream_t st) {   \
    return launch_fields_t<S, R>(src, g, P, rho, u, gd, st);                                  \
  }                                                                                           \
  cudaError_t launch_collide_nodes_##SUFFIX(const PhysParams& P, const double* fin,           \
                                            double* fout, double* rho, double* u, double* gd, \
                                            int64_t M, cudaStream_t st) {                     \
    return launch_collide_nodes_t<S, R>(P, fin, fout, rho, u, gd, M, st);                     \
  }                                                                                           \
  cudaError_t launch_export_##SUFFIX(const void* src, const Geom& g, double rho0,             \
                                     double inv_scale, double* out, cudaStream_t st) {        \
    return launch_export_t<S>(src, g, rho0, inv_scale, out, st);                              \
  }                                                                                           \
  cudaError_t launch_omega_nodes_##SUFFIX(const PhysParams& P, const double* rho,             \
                                          const double* m, double* omega, double* gd,         \
                                          int64_t M, cudaStream_t st) {                       \
    return launch_omega_nodes_t<R>(P, rho, m, omega, gd, M, st);                              \
  }                                                                                           \
  cudaError_t launch_import_##SUFFIX(const double* in, const Geom& g, double rho0,            \
                                     double inv_scale, void* dst, cudaStream_t st) {          \
    return launch_import_t<S>(in, g, rho0, inv_scale, dst, st);                               \
  }                                                                                           \
  }
