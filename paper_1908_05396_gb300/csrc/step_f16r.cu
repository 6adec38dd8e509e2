// step_f16r.cu -- kernels of the F16R storage form: FP16 populations stored
// relative to the writing node's first-order equilibrium.
//
// The deviations are carried scaled by lam = 1024 (as in the F16S form, with
// the factor folded into the collision's constants).  Each node keeps a
// reference (lam (rho - rho0), lam 3 rho u) of its last collision as four
// FP16 values next to its populations, and stores
//     s_q = fp16( lam ( f~_q - w_q rho0 ) - r_q ),
//     r_q = w_q [ dr + e_q . v ],  (dr, v) the reference,
// which removes the rest value and the first-order (velocity) part of the
// equilibrium, the largest parts of f~, before FP16 rounding (stochastic in
// the step kernels, see enc16_sr2).  A reader decodes with the reference of
// the node that wrote the value: the upwind neighbour for a streamed value,
// itself for a bounced one.  Both sides use the reference exactly as stored,
// so decoding undoes the encoding up to the FP16 rounding of the small
// remainder (and one FP32 rounding).  A reference is read by 19 readers, one
// 64-bit load each: in FP16 the 19 loads of a node need half the registers in
// flight (and half the L1/L2 traffic) of FP32 references.
// The reference arrays are double-buffered with the populations.
#include "batch.cuh"
#include "sround.cuh"

namespace clbm {
namespace {

// The back-transform of the collision: unforced, the populations are rebuilt
// from the pair values (the inputs die early, which frees registers; the FP16
// rounding noise of the stores lies far above the FP32 roundings of the
// rebuild); with a body force, one correction per population, which keeps a
// weak force's increments to one rounding (rebuilt from the pairs, a forced
// channel's velocity drifted by 1e-3 against FP64).
constexpr int LOG2LAM = 10;  // log2 of the scale of the carried deviations
constexpr float LAM = float(1 << LOG2LAM);
static_assert(double(1 << LOG2LAM) == F16_SCALE, "one FP16 storage scale");

// The reference of a node with density rho = rho0 + drho and velocity u,
// rounded to FP16 for storage; r receives the rounded values.
__device__ __forceinline__ uint2 ref_make(float drho, float rho, float ux, float uy, float uz,
                                          RefT<float>& r) {
  const float r3 = mulr(3.0f * LAM, rho);
  const __half2 a = __floats2half2_rn(mulr(LAM, drho), mulr(r3, ux)),
                b = __floats2half2_rn(mulr(r3, uy), mulr(r3, uz));
  const float2 fa = __half22float2(a), fb = __half22float2(b);
  r = {fa.x, fa.y, fb.x, fb.y};
  uint2 v;
  v.x = *reinterpret_cast<const unsigned*>(&a);
  v.y = *reinterpret_cast<const unsigned*>(&b);
  return v;
}

__device__ __forceinline__ float dec16(__half v) { return __half2float(v); }
__device__ __forceinline__ __half enc16(float v) { return __float2half_rn(v); }

// v plus (sgn = 1) or minus (sgn = -1) the first-order equilibrium deviation
// of direction q about the reference, lam w_q [drho + 3 rho (e_q . u)],
// with the weights ref_wt.
__device__ __forceinline__ float plus_ref(float v, int q, const RefT<float>& r, float sgn = 1.0f) {
  return fma(sgn * ref_wt(q), ref_sum(q, r), v);
}

struct RefArgs {
  const uint2* refq[Q];  // refq[q][i]: reference of the upwind neighbour of node i
  const uint2* ref_src;  // references of the source step
  uint2* ref_dst;        // references written by this step
  StepSeed seed;         // the lattice's steps done before this one
};

// Pull of all 19 directions into node (x, y, z) with index i, for a node on
// any face, by the face rules of pull_face; each value is decoded with the
// reference of the node that wrote it: the upwind (or wrapped) node for a
// streamed value, the node itself for a bounced one.
__device__ __forceinline__ void pull_face_ref(const __half* __restrict__ src,
                                              const uint2* __restrict__ ref, int64_t qstride,
                                              int nx, int ny, int nz, int pitch, int plane,
                                              unsigned fb, int x, int y, int z, int i,
                                              const float* lidc, float (&d)[Q]) {
  const Faces f = faces_of(x, y, z, nx, ny, nz, pitch, plane, fb);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const bool bounce = (f.wall & up_faces(q)) != 0;
    const int j = bounce ? i : i - (cz(q) * plane + cy(q) * pitch + cx(q)) + up_wrap(f, q);
    const __half v = (src + (bounce ? int64_t(opp(q)) * qstride : int64_t(q) * qstride))[j];
    // a bounced value is decoded as opp(q): e_q . v changes sign
    const float sgn = bounce ? -1.0f : 1.0f;
    RefT<float> t = ref1(ref + j);
    t = {t.dr, mulr(sgn, t.vx), mulr(sgn, t.vy), mulr(sgn, t.vz)};
    d[q] = plus_ref(dec16(v), q, t);
    if (f.lid & up_faces(q)) d[q] += lidc[q];
  }
}

// Pull of node (x, y, z) with index i: warps off every face load directly.
__device__ __forceinline__ void pull_node_ref(const StepArgs<__half, float>& a, const RefArgs& r,
                                              int x, int y, int z, int i, float (&d)[Q]) {
  const bool inner = y > 0 && y < a.ny - 1 && z > 0 && z < a.nz - 1 && x > 0 && x < a.nx - 1;
  if (__all_sync(__activemask(), inner)) {
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = plus_ref(dec16(a.srcq[q][i]), q, ref1(r.refq[q] + i));
  } else {
    pull_face_ref(a.src, r.ref_src, a.qstride, a.nx, a.ny, a.nz, a.pitch, a.plane, a.facebits, x,
                  y, z, i, a.lidc, d);
  }
}

// Collide the node and store it (as collide_pair and store_pair).
template <bool FORCE, bool UNIT>
__device__ __forceinline__ void collide_store_ref(const StepArgs<__half, float>& a,
                                                  const RefArgs& r, int i, unsigned step,
                                                  float (&d)[Q], NodeOut<float>& o) {
  auto reference = [&](const NodeOut<float>& n) {
    RefT<float> t;
    r.ref_dst[i] = ref_make(n.rho - a.C.rho0, n.rho, n.ux, n.uy, n.uz, t);
    return t;
  };
  if constexpr (UNIT && !FORCE) {
    collide_unit<float, false, true, LOG2LAM>(a.C, d, o, reference);
  } else {
    collide<float, FORCE, !FORCE, LOG2LAM, UNIT>(a.C, d, o);
    const RefT<float> t = reference(o);
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = plus_ref(d[q], q, t, -1.0f);
  }
  store_sr1([&](int q) { return a.dstq[q] + i; }, d, uint32_t(i), step);
}

// One node per thread.
template <bool FORCE, bool CHECK, bool UNIT>
__global__ void __launch_bounds__(256) step_ref_kernel(const StepArgs<__half, float> a,
                                                       const RefArgs r) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = a.zrev ? a.nz - 1 - int(blockIdx.z) : int(blockIdx.z);  // as step_kernel
  const bool active = x < a.nx && y < a.ny;
  if (!CHECK && !active) return;
  CheckSums sums;
  if (active) {
    const int i = z * a.plane + y * a.pitch + x;
    float d[Q];
    pull_node_ref(a, r, x, y, z, i, d);
    NodeOut<float> o;
    collide_store_ref<FORCE, UNIT>(a, r, i, r.seed.get(), d, o);
    if (CHECK)
      check_node(sums, o.rho, o.ux, o.uy, o.uz, a.C.rho0, static_cast<float*>(a.cb.uprev) + i,
                 int64_t(a.plane) * a.nz);
  }
  if (CHECK) block_sums(sums, check_row(a.cb), a.cb.flag);
}

template <bool FORCE>
__global__ void __launch_bounds__(256) fields_ref_kernel(const StepArgs<__half, float> a,
                                                         const RefArgs r, const FieldsOut f) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= a.nx || y >= a.ny) return;
  float d[Q];
  pull_node_ref(a, r, x, y, z, z * a.plane + y * a.pitch + x, d);
  NodeOut<float> o;
  node_fields<float, FORCE, LOG2LAM>(a.C, d, f.gd != nullptr, o);
  write_fields(f, o, a.nx, a.ny, a.nz, x, y, z);
}

__global__ void export_ref_kernel(const __half* __restrict__ src, const uint2* __restrict__ ref,
                                  Geom g, float rho0, double* __restrict__ out) {
  const int64_t N = int64_t(g.nx) * g.ny * g.nz;
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= N * Q) return;
  const int q = int(t / N);
  const int64_t k = t - int64_t(q) * N;
  const int x = int(k % g.nx), y = int((k / g.nx) % g.ny), z = int(k / (int64_t(g.nx) * g.ny));
  const int64_t i = int64_t(z) * g.plane + int64_t(y) * g.pitch + x;
  const float dev = plus_ref(dec16(src[q * g.qstride + i]), q, ref1(ref + i));
  out[t] = double(dev) * (1.0 / double(LAM)) + wt<double>(q) * double(rho0);
}

// One thread per node: the reference is the node's own moments of the
// imported populations.
__global__ void import_ref_kernel(const double* __restrict__ in, Geom g, float rho0,
                                  __half* __restrict__ dst, uint2* __restrict__ ref) {
  const int64_t N = int64_t(g.nx) * g.ny * g.nz;
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= N) return;
  const int x = int(k % g.nx), y = int((k / g.nx) % g.ny), z = int(k / (int64_t(g.nx) * g.ny));
  const int64_t i = int64_t(z) * g.plane + int64_t(y) * g.pitch + x;
  double f[Q], rho = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    f[q] = in[q * N + k];
    rho += f[q];
    jx += cx(q) * f[q];
    jy += cy(q) * f[q];
    jz += cz(q) * f[q];
  }
  RefT<float> rr;
  ref[i] = ref_make(float(rho - rho0), float(rho), float(jx / rho), float(jy / rho),
                    float(jz / rho), rr);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    dst[q * g.qstride + i] =
        enc16(plus_ref(float((f[q] - wt<double>(q) * rho0) * double(LAM)), q, rr, -1.0f));
}

// M independent nodes: store (with its own reference), load, collide, store
// again with the new reference, load.
template <bool FORCE>
__global__ void collide_nodes_ref_kernel(CollideConst<float> C, const double* __restrict__ fin,
                                         double* __restrict__ fout, double* rho, double* u,
                                         double* gd, int64_t M) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= M) return;
  const float rho0 = C.rho0;
  double r0 = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const double v = fin[q * M + k];
    r0 += v;
    jx += cx(q) * v;
    jy += cy(q) * v;
    jz += cz(q) * v;
  }
  RefT<float> rr;
  ref_make(float(r0 - rho0), float(r0), float(jx / r0), float(jy / r0), float(jz / r0), rr);
  float d[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float dev = float((fin[q * M + k] - wt<double>(q) * rho0) * double(LAM));
    d[q] = plus_ref(dec16(enc16(plus_ref(dev, q, rr, -1.0f))), q, rr);
  }
  NodeOut<float> o;
  collide<float, FORCE, !FORCE, LOG2LAM, true>(C, d, o);
  ref_make(o.rho - rho0, o.rho, o.ux, o.uy, o.uz, rr);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float dev = plus_ref(dec16(enc16(plus_ref(d[q], q, rr, -1.0f))), q, rr);
    fout[q * M + k] = double(dev) * (1.0 / double(LAM)) + wt<double>(q) * double(rho0);
  }
  if (rho) rho[k] = double(o.rho);
  if (u) {
    u[k] = double(o.ux);
    u[M + k] = double(o.uy);
    u[2 * M + k] = double(o.uz);
  }
  if (gd) gd[k] = double(o.gamma_dot);
}

RefArgs ref_args(const void* ref_src, void* ref_dst, const Geom& g, StepSeed seed) {
  RefArgs r;
  r.seed = seed;
  r.ref_src = static_cast<const uint2*>(ref_src);
  r.ref_dst = static_cast<uint2*>(ref_dst);
  for (int q = 0; q < Q; ++q) {
    const int64_t off = int64_t(cz(q)) * g.plane + int64_t(cy(q)) * g.pitch + cx(q);
    r.refq[q] = reinterpret_cast<const uint2*>(reinterpret_cast<uintptr_t>(ref_src) -
                                                off * int64_t(sizeof(uint2)));
  }
  return r;
}

}  // namespace

// One node of the batched step in the F16R form: the same pull, references
// and collision as step_ref_kernel.
template <bool FORCE>
__device__ void batch_node_ref(const LatDesc<float>& L, int parity, int x, int y, int z,
                               unsigned step, NodeOut<float>& o) {
  const __half* src = static_cast<const __half*>(L.buf[parity]);
  __half* dst = static_cast<__half*>(const_cast<void*>(L.buf[parity ^ 1]));
  const uint2* rs = static_cast<const uint2*>(L.ref[parity]);
  uint2* rd = static_cast<uint2*>(const_cast<void*>(L.ref[parity ^ 1]));
  const float rho0 = L.C.rho0;
  const int qs = int(L.qstride), plane = L.plane, pitch = L.pitch;
  const int i = z * plane + y * pitch + x;
  float d[Q];
  const bool inner = y > 0 && y < L.ny - 1 && z > 0 && z < L.nz - 1 && x > 0 && x < L.nx - 1;
  if (__all_sync(__activemask(), inner)) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int up = i - (cz(q) * plane + cy(q) * pitch + cx(q));
      d[q] = plus_ref(dec16(src[q * qs + up]), q, ref1(rs + up));
    }
  } else {
    pull_face_ref(src, rs, L.qstride, L.nx, L.ny, L.nz, pitch, plane, L.facebits, x, y, z, i,
                  L.lidc, d);
  }
  collide<float, FORCE, !FORCE, LOG2LAM, false>(L.C, d, o);
  RefT<float> rr;
  rd[i] = ref_make(o.rho - rho0, o.rho, o.ux, o.uy, o.uz, rr);
#pragma unroll
  for (int q = 0; q < Q; ++q) d[q] = plus_ref(d[q], q, rr, -1.0f);
  store_sr1([&](int q) { return dst + (q * qs + i); }, d, uint32_t(i), step);
}

cudaError_t launch_step_f16r(const void* src, void* dst, const void* ref_src, void* ref_dst,
                             const Geom& g, const PhysParams& P, const CheckBufs& cb, bool check,
                             dim3 block, int64_t step, const unsigned* base, cudaStream_t st) {
  const StepArgs<__half, float> a = step_args<__half, float>(src, dst, g, P, cb);
  const uint2* rs = static_cast<const uint2*>(ref_src);
  uint2* rd = static_cast<uint2*>(ref_dst);
  const StepSeed seed{unsigned(uint64_t(step)), base};
  const bool unit = unit_rates(P);
  if (unit && pair_pays(g, true))
    return launch_step_pair<PAIR_REF>(a, PairExtra{rs, rd, seed},
                                      P.has_force != 0, check, block, st);
  const RefArgs r = ref_args(rs, rd, g, seed);
  const dim3 grid((g.nx + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y, g.nz);
  void (*kernel)(const StepArgs<__half, float>, const RefArgs) = nullptr;
#define CLBM_REF(F, C_) kernel = unit ? step_ref_kernel<F, C_, true> : step_ref_kernel<F, C_, false>
  if (P.has_force) {
    if (check) CLBM_REF(true, true);
    else CLBM_REF(true, false);
  } else {
    if (check) CLBM_REF(false, true);
    else CLBM_REF(false, false);
  }
#undef CLBM_REF
  return pdl_launch(kernel, grid, block, st, a, r);
}

cudaError_t launch_fields_f16r(const void* src, const void* ref, const Geom& g,
                               const PhysParams& P, double* rho, double* u, double* gd,
                               cudaStream_t st) {
  const dim3 block(32, 4);
  const dim3 grid((g.nx + 31) / 32, (g.ny + 3) / 4, g.nz);
  const StepArgs<__half, float> a = step_args<__half, float>(src, nullptr, g, P, CheckBufs{});
  const RefArgs r = ref_args(static_cast<const uint2*>(ref), nullptr, g, StepSeed{});
  const FieldsOut f{rho, u, gd};
  if (P.has_force) fields_ref_kernel<true><<<grid, block, 0, st>>>(a, r, f);
  else fields_ref_kernel<false><<<grid, block, 0, st>>>(a, r, f);
  return cudaGetLastError();
}

cudaError_t launch_export_f16r(const void* src, const void* ref, const Geom& g, double rho0,
                               double* out, cudaStream_t st) {
  const int64_t total = int64_t(g.nx) * g.ny * g.nz * Q;
  const int b = 256;
  export_ref_kernel<<<unsigned((total + b - 1) / b), b, 0, st>>>(
      static_cast<const __half*>(src), static_cast<const uint2*>(ref), g, float(rho0), out);
  return cudaGetLastError();
}

cudaError_t launch_import_f16r(const double* in, const Geom& g, double rho0, void* dst, void* ref,
                               cudaStream_t st) {
  const int64_t N = int64_t(g.nx) * g.ny * g.nz;
  const int b = 128;
  import_ref_kernel<<<unsigned((N + b - 1) / b), b, 0, st>>>(in, g, float(rho0),
                                                              static_cast<__half*>(dst),
                                                              static_cast<uint2*>(ref));
  return cudaGetLastError();
}

cudaError_t launch_collide_nodes_f16r(const PhysParams& P, const double* fin, double* fout,
                                      double* rho, double* u, double* gd, int64_t M,
                                      cudaStream_t st) {
  const int b = 128;
  const unsigned grid = unsigned((M + b - 1) / b);
  const CollideConst<float> C = make_const<float>(P, double(LAM));
  if (P.has_force) collide_nodes_ref_kernel<true><<<grid, b, 0, st>>>(C, fin, fout, rho, u, gd, M);
  else collide_nodes_ref_kernel<false><<<grid, b, 0, st>>>(C, fin, fout, rho, u, gd, M);
  return cudaGetLastError();
}

}  // namespace clbm

CLBM_DEFINE_BATCH(f16r, __half, float, true)
