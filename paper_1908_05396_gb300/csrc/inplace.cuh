// inplace.cuh -- the fused step with ONE population buffer (in-place
// streaming), for the FP64, FP32 and F16S forms.
//
// Two kinds of step alternate, and the buffer A[q][node] holds one of two
// layouts between steps:
//   layout 0 ("swapped"): A[opp(q)][x] = f~_q(x), the post-collision value of
//       node x in direction q kept in its opposite slot;
//   layout 1 ("streamed"): A[q][x] = f~_q(x - e_q), the value node x pulls in
//       direction q (or, where x - e_q is beyond a wall or the lid, the
//       bounced value f~_opp(q)(x)).
// A neighbour step (layout 0 -> 1) reads f_q(x) from A[opp(q)][x - e_q],
// collides and writes f~_q(x) to A[q][x + e_q]; a local step (layout 1 -> 0)
// reads A[q][x], collides and writes f~_q(x) to A[opp(q)][x].  In both, the
// 19 slots a node reads are exactly the 19 it writes, so one thread per node
// updates the buffer in place with no race.  Walls and the lid follow the
// pull rules of the two-buffer step (pull_face): a value whose source or
// destination crosses a non-periodic face stays at the node in the opposite
// slot (halfway bounce-back), the lid term 6 w_q rho0 (e_q . U) is added when
// it is read (so stored values are the exact post-collision ones), and
// periodic faces wrap.  Every step computes exactly what the two-buffer step
// computes, with the same bytes per update and half the memory.
#pragma once

namespace clbm {

// Pre-collision values of node i in layout L (any node, faces included).  As
// in pull_face the face rules select addresses.
template <typename S, typename R, int L>
__device__ __forceinline__ void aa_read(const S* A, int64_t qs, int i, int pitch, int plane,
                                        const Faces& f, const R* lidc, R (&d)[Q]) {
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    // streamed layout: the own slot; swapped layout: the upwind node's
    // opposite slot, or the own slot q (bounce: f~_opp(q)(x) sits in slot
    // opp(opp(q)) = q)
    const bool own = L == 1 || (f.wall & up_faces(q)) != 0;
    const int j = i - (cz(q) * plane + cy(q) * pitch + cx(q)) + up_wrap(f, q);
    const S* p = A + (own ? int64_t(q) * qs : int64_t(opp(q)) * qs);
    d[q] = Codec<S, R>::dec(p[own ? i : j], R(1));
    if (f.lid & up_faces(q)) d[q] += lidc[q];  // (a lid always bounces)
  }
}

// Post-collision values of node i written for the next layout: after a
// neighbour step (layout 1) to the downstream node's slot q, or back into
// the own opposite slot where the downstream side crosses a wall or the lid.
template <typename S, typename R>
__device__ __forceinline__ void aa_write_streamed(S* A, int64_t qs, int i, int pitch, int plane,
                                                  const Faces& f, const R (&d)[Q]) {
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const bool bounce = (f.wall & up_faces(opp(q))) != 0;
    const int j = i + (cz(q) * plane + cy(q) * pitch + cx(q)) + up_wrap(f, opp(q));
    S* p = A + (bounce ? int64_t(opp(q)) * qs : int64_t(q) * qs);
    p[bounce ? i : j] = Codec<S, R>::enc(d[q], R(1));
  }
}

// In-place update of node (x, y, z) with index i.  LIN is the layout the step
// reads: 0 -> neighbour step (srcq[q] = A + opp(q) qs - off(q), dstq[q] =
// A + q qs + off(q)), 1 -> local step (srcq[q] = A + q qs, dstq[q] = A +
// opp(q) qs); a.src is the buffer A.  Nodes off the faces take the direct path.
template <typename S, typename R, int LIN, bool FORCE, bool UNIT>
__device__ __forceinline__ void aa_update(const StepArgs<S, R>& a, int x, int y, int z, int i,
                                          NodeOut<R>& o) {
  S* A = const_cast<S*>(a.src);
  const bool inner = x > 0 && x < a.nx - 1 && y > 0 && y < a.ny - 1 && z > 0 && z < a.nz - 1;
  const Faces f = faces_of(x, y, z, a.nx, a.ny, a.nz, a.pitch, a.plane, a.facebits);
  R d[Q];
  if (inner) {
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = Codec<S, R>::dec(a.srcq[q][i], R(1));
  } else {
    aa_read<S, R, LIN>(A, a.qstride, i, a.pitch, a.plane, f, a.lidc, d);
  }
  collide<R, FORCE, pair_out<S>(), log2_scale<S>(), UNIT>(a.C, d, o);
  if (LIN == 1 || inner) {
#pragma unroll
    for (int q = 0; q < Q; ++q) a.dstq[q][i] = Codec<S, R>::enc(d[q], R(1));
  } else {
    aa_write_streamed<S, R>(A, a.qstride, i, a.pitch, a.plane, f, d);
  }
}

// One in-place step.  UNIT as in step_kernel, but that the FP32-math forms have
// the register-capped variant with other rates too: 128^3 FP32 in blocks of 32 x 8
// 70.3 us a step against 76.2 uncapped, tuned 63.8 against 64.9 (F16S tuned 54.8
// against 56.2).
template <typename S, typename R, int LIN, bool FORCE, bool CHECK, bool CAP, bool UNIT>
__global__ void __launch_bounds__(256, CAP ? 4 : 1) step_aa_kernel(const StepArgs<S, R> a) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  const bool active = x < a.nx && y < a.ny;
  if (!CHECK && !active) return;
  CheckSums sums;
  if (active) {
    const int i = z * a.plane + y * a.pitch + x;
    NodeOut<R> o;
    aa_update<S, R, LIN, FORCE, UNIT>(a, x, y, z, i, o);
    if (CHECK)
      check_node(sums, o.rho, o.ux, o.uy, o.uz, a.C.rho0, static_cast<R*>(a.cb.uprev) + i,
                 int64_t(a.plane) * a.nz);
  }
  if (CHECK) block_sums(sums, check_row(a.cb), a.cb.flag);
}

// rho, u and |gamma_dot| of the next collision, from either layout.
template <typename S, typename R, int L, bool FORCE>
__global__ void __launch_bounds__(256) fields_aa_kernel(const StepArgs<S, R> a,
                                                        const FieldsOut f) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= a.nx || y >= a.ny) return;
  const int i = z * a.plane + y * a.pitch + x;
  R d[Q];
  aa_read<S, R, L>(a.src, a.qstride, i, a.pitch, a.plane,
                   faces_of(x, y, z, a.nx, a.ny, a.nz, a.pitch, a.plane, a.facebits), a.lidc, d);
  NodeOut<R> o;
  node_fields<R, FORCE, log2_scale<S>()>(a.C, d, f.gd != nullptr, o);
  write_fields(f, o, a.nx, a.ny, a.nz, x, y, z);
}

// The post-collision populations f~_q(x) (the state the two-buffer form
// stores), from either layout: layout 0 holds them in the opposite slots;
// layout 1 holds them at the downstream node, or at the node itself in the
// opposite slot where the downstream side is a wall or the lid.
template <typename S>
__global__ void __launch_bounds__(128) export_aa_kernel(const S* __restrict__ A, Geom g,
                                                        double rho0, double inv_scale, int layout,
                                                        double* __restrict__ out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  const int64_t N = int64_t(g.nx) * g.ny * g.nz, k = (int64_t(z) * g.ny + y) * g.nx + x;
  const int pitch = g.pitch, plane = int(g.plane), i = z * plane + y * pitch + x;
  const Faces f = faces_of(x, y, z, g.nx, g.ny, g.nz, pitch, plane, g.facebits);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    // the opposite slot: layout 0, or a value bounced downstream
    const bool own = layout == 0 || (f.wall & up_faces(opp(q))) != 0;
    const int j = i + (cz(q) * plane + cy(q) * pitch + cx(q)) + up_wrap(f, opp(q));
    const S v = (A + (own ? opp(q) : q) * g.qstride)[own ? i : j];
    out[q * N + k] =
        double(Codec<S, double>::dec(v, inv_scale)) * inv_scale + wt<double>(q) * rho0;
  }
}

// Import a state f~ into layout 0.
template <typename S>
__global__ void __launch_bounds__(128) import_aa_kernel(const double* __restrict__ in, Geom g,
                                                        double rho0, double scale,
                                                        S* __restrict__ A) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  const int64_t N = int64_t(g.nx) * g.ny * g.nz, k = (int64_t(z) * g.ny + y) * g.nx + x;
  const int64_t i = int64_t(z) * g.plane + int64_t(y) * g.pitch + x;
#pragma unroll
  for (int q = 0; q < Q; ++q)
    A[opp(q) * g.qstride + i] =
        Codec<S, double>::enc((in[q * N + k] - wt<double>(q) * rho0) * scale, scale);
}

// ---- host-side launchers ------------------------------------------------------
// The arguments of a step that reads layout `layout` (all planes in ascending
// order: an alternating sweep, either parity, measured 2 % slower here).
template <typename S, typename R>
StepArgs<S, R> aa_args(void* buf, const Geom& g, const PhysParams& P, const CheckBufs& cb,
                       int layout) {
  StepArgs<S, R> a = step_args<S, R>(buf, buf, g, P, cb);
  const uintptr_t base = reinterpret_cast<uintptr_t>(buf);
  for (int q = 0; q < Q; ++q) {
    const int64_t off = int64_t(cz(q)) * g.plane + int64_t(cy(q)) * g.pitch + cx(q);
    // address arithmetic through integers: a shifted base may lie outside the
    // buffer; only base + i of a node whose partner node exists is used
    const int64_t sq = layout == 0 ? int64_t(opp(q)) * g.qstride - off : int64_t(q) * g.qstride;
    const int64_t dq = layout == 0 ? int64_t(q) * g.qstride + off : int64_t(opp(q)) * g.qstride;
    a.srcq[q] = reinterpret_cast<const S*>(base + sq * int64_t(sizeof(S)));
    a.dstq[q] = reinterpret_cast<S*>(base + dq * int64_t(sizeof(S)));
  }
  return a;
}

template <typename S, typename R>
cudaError_t launch_step_aa_t(void* buf, const Geom& g, const PhysParams& P, const CheckBufs& cb,
                             bool check, dim3 block, int npt, int layout, cudaStream_t st) {
  const StepArgs<S, R> a = aa_args<S, R>(buf, g, P, cb, layout);
  const bool cap = (npt & 4) != 0;
  const dim3 grid((g.nx + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y, g.nz);
  const bool unit = unit_rates(P);
  constexpr bool RC = !std::is_same<R, double>::value;
  void (*kernel)(const StepArgs<S, R>) = nullptr;
#define CLBM_AA(L, F, C_)                                                     \
  kernel = unit && cap ? step_aa_kernel<S, R, L, F, C_, true, true>           \
           : unit      ? step_aa_kernel<S, R, L, F, C_, false, true>          \
           : cap       ? step_aa_kernel<S, R, L, F, C_, RC, false>            \
                       : step_aa_kernel<S, R, L, F, C_, false, false>
  if (layout == 0) {
    if (P.has_force) { if (check) CLBM_AA(0, true, true); else CLBM_AA(0, true, false); }
    else { if (check) CLBM_AA(0, false, true); else CLBM_AA(0, false, false); }
  } else {
    if (P.has_force) { if (check) CLBM_AA(1, true, true); else CLBM_AA(1, true, false); }
    else { if (check) CLBM_AA(1, false, true); else CLBM_AA(1, false, false); }
  }
#undef CLBM_AA
  return pdl_launch(kernel, grid, block, st, a);
}

template <typename S, typename R>
cudaError_t launch_fields_aa_t(const void* buf, const Geom& g, const PhysParams& P, int layout,
                               double* rho, double* u, double* gd, cudaStream_t st) {
  const dim3 block(32, 4);
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  const StepArgs<S, R> a = step_args<S, R>(buf, nullptr, g, P, CheckBufs{});
  const FieldsOut f{rho, u, gd};
  if (layout == 0) {
    if (P.has_force) fields_aa_kernel<S, R, 0, true><<<grid, block, 0, st>>>(a, f);
    else fields_aa_kernel<S, R, 0, false><<<grid, block, 0, st>>>(a, f);
  } else {
    if (P.has_force) fields_aa_kernel<S, R, 1, true><<<grid, block, 0, st>>>(a, f);
    else fields_aa_kernel<S, R, 1, false><<<grid, block, 0, st>>>(a, f);
  }
  return cudaGetLastError();
}

template <typename S>
cudaError_t launch_export_aa_t(const void* buf, const Geom& g, double rho0, double inv_scale,
                               int layout, double* out, cudaStream_t st) {
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  export_aa_kernel<S><<<grid, dim3(32, 4), 0, st>>>(static_cast<const S*>(buf), g, rho0,
                                                    inv_scale, layout, out);
  return cudaGetLastError();
}

template <typename S>
cudaError_t launch_import_aa_t(const double* in, const Geom& g, double rho0, double inv_scale,
                               void* buf, cudaStream_t st) {
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  import_aa_kernel<S><<<grid, dim3(32, 4), 0, st>>>(in, g, rho0, 1.0 / inv_scale,
                                                    static_cast<S*>(buf));
  return cudaGetLastError();
}

}  // namespace clbm

// Defines the in-place launchers of launch.h for storage type S, math type R.
#define CLBM_DEFINE_AA(SUFFIX, S, R)                                                           \
  namespace clbm {                                                                             \
  cudaError_t launch_step_aa_##SUFFIX(void* buf, const Geom& g, const PhysParams& P,           \
                                      const CheckBufs& cb, bool check, dim3 block, int npt,    \
                                      int layout, cudaStream_t st) {                           \
    return launch_step_aa_t<S, R>(buf, g, P, cb, check, block, npt, layout, st);               \
  }                                                                                            \
  cudaError_t launch_fields_aa_##SUFFIX(const void* buf, const Geom& g, const PhysParams& P,   \
                                        int layout, double* rho, double* u, double* gd,        \
                                        cudaStream_t st) {                                     \
    return launch_fields_aa_t<S, R>(buf, g, P, layout, rho, u, gd, st);                        \
  }                                                                                            \
  cudaError_t launch_export_aa_##SUFFIX(const void* buf, const Geom& g, double rho0,           \
                                        double inv_scale, int layout, double* out,             \
                                        cudaStream_t st) {                                     \
    return launch_export_aa_t<S>(buf, g, rho0, inv_scale, layout, out, st);                    \
  }                                                                                            \
  cudaError_t launch_import_aa_##SUFFIX(const double* in, const Geom& g, double rho0,          \
                                        double inv_scale, void* buf, cudaStream_t st) {        \
    return launch_import_aa_t<S>(in, g, rho0, inv_scale, buf, st);                             \
  }                                                                                            \
  }
