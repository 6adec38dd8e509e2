// pair.cuh -- the FP16 storage forms stepped two nodes per thread.
//
// A thread owns the nodes x and x + 1 (x even) of a row and collides them as
// one packed pair (V2).  Why pairs along x:
//   - FP16 forms move half the bytes of FP32, so instruction issue bounds
//     them, not HBM; packed FP32 instructions issue once for two nodes (a
//     packed multiply-add issues in one slot and takes the FP32 pipe for 2.1
//     cycles a warp, where two scalar ones of three register operands take
//     3.8), and index and face logic is shared by two nodes;
//   - the two values of a direction with e_x = 0, and every stored value,
//     are one aligned 32-bit access and one conversion instruction.
// Rows y and y + 1 as the pair (the first attempt, for FP32 too) keep every
// 16-bit access and lose most of this.
// Measured, one node per thread -> pairs, us a step: F16S 323 -> 233 on 256^3
// (5.5 TB/s) and 49.8 -> 38.6 on 128^3; F16R 753 -> 418 and 95 -> 61, whose
// 19 reference loads a node become 9.5 and whose reference terms are packed.
// DRAM latency and the drain between dependent steps bound it now (128^3:
// issue slots 49 % busy).
//
// Included by kernels.cuh (StepArgs, codecs, pdl_launch).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "sround.cuh"

namespace clbm {

__device__ __forceinline__ V2 ld2(const __half* p) {  // p even: one 32-bit load
  return V2(__half22float2(*reinterpret_cast<const __half2*>(p)));
}
__device__ __forceinline__ float ld1(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ void set0(V2& v, float f) { v.v.x = f; }
__device__ __forceinline__ void set1(V2& v, float f) { v.v.y = f; }

// ---- F16R references -----------------------------------------------------
// (dr, v) of a node: lam (rho - rho0) and lam 3 rho u, as stored (FP16).
template <typename R>
struct RefT {
  R dr, vx, vy, vz;
};
__device__ __forceinline__ RefT<float> ref_dec(uint2 v) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
  return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ RefT<float> ref1(const uint2* p) { return ref_dec(*p); }
// dr + e_q . v, the part of the reference term that w_q multiplies; the sums
// are associated alike for a node and a pair, so that a reader forms the
// value the writer subtracted.
template <typename R>
__device__ __forceinline__ R ref_sum(int q, const RefT<R>& r) {
  R s = r.dr;
  if (cy(q) == 1) s = s + r.vy;
  if (cy(q) == -1) s = s - r.vy;
  if (cz(q) == 1) s = s + r.vz;
  if (cz(q) == -1) s = s - r.vz;
  if (cx(q) == 1) s = s + r.vx;
  if (cx(q) == -1) s = s - r.vx;
  return s;
}

// ---- pull ----------------------------------------------------------------
// Where a pair's upwind values are, for the lone step (precomputed base
// pointers of StepArgs) and the batch (offsets from the lattice's buffer):
//   up(q): upwind value of the pair's first node; own(q): the pair's own
//   value; ref: the pair's own F16R reference.
struct LonePair {
  const StepArgs<__half, float>& a;
  const uint2* ref;
  int i;
  __device__ __forceinline__ const __half* up(int q) const { return a.srcq[q] + i; }
  __device__ __forceinline__ const __half* own(int q) const {
    return a.src + int64_t(q) * a.qstride + i;
  }
  __device__ __forceinline__ int nx() const { return a.nx; }
  __device__ __forceinline__ int ny() const { return a.ny; }
  __device__ __forceinline__ int nz() const { return a.nz; }
  __device__ __forceinline__ int pitch() const { return a.pitch; }
  __device__ __forceinline__ int plane() const { return a.plane; }
  __device__ __forceinline__ unsigned faces() const { return a.facebits; }
  __device__ __forceinline__ float lid(int q) const { return a.lidc[q]; }
};

// One direction of one node that crosses an x face (and no y or z wall):
// the periodic wrap (dx nodes along x from the node's plain upwind value at
// u, reference at r), or halfway bounce-back from the node's own opposite
// value, plus the lid term.
template <bool REF, typename P>
__device__ __forceinline__ float xface_value(const P& p, int q, int k, int n, const __half* u,
                                             const uint2* r, int dx) {
  if (k == BC_PERIODIC) {
    float v = ld1(u + dx);
    if (REF) v = fma(wt<float>(q), ref_sum(q, ref1(r + dx)), v);
    return v;
  }
  float v = ld1(p.own(opp(q)) + n);
  if (REF) v = fma(wt<float>(q), ref_sum(opp(q), ref1(p.ref + n)), v);
  return k == BC_LID ? v + p.lid(q) : v;
}

// The pre-collision deviations of the pair (x, x + 1) in row (y, z).  Rows off
// the y and z faces load every direction unconditionally and then replace, in
// the threads that hold x = 0 or x = nx - 1, the five directions that come
// from outside; rows on a y or z face resolve each direction.  When nx is odd
// the last pair's second node lies in the row's padding: it is computed from
// whatever is there and stored there.
template <bool REF, typename P>
__device__ __forceinline__ void pull_pair(const P& p, int x, int y, int z, V2 (&d)[Q]) {
  const int nx = p.nx(), pitch = p.pitch(), plane = p.plane();
  const unsigned fb = p.faces();
  const int kl = int(fb & 3u), kr = int((fb >> 2) & 3u);
  const bool first = x == 0, last = x + 2 >= nx;   // the pair holds x = 0 / x = nx - 1
  const int nr = nx - 1 - x;                        // which node is at nx - 1
  if (y > 0 && y < p.ny() - 1 && z > 0 && z < p.nz() - 1) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const __half* u = p.up(q);
      if (cx(q) == 0) d[q] = ld2(u);
      else d[q] = V2(ld1(u), ld1(u + 1));
    }
    if (REF) {
      // Columns of upwind nodes (e_y, e_z), each one 128-bit reference load
      // for the pair's own x and, where the column's directions have e_x != 0,
      // a 64-bit load on either side.
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        if (cx(c) != 0) continue;
        const uint2* rc = p.ref - (cz(c) * plane + cy(c) * pitch);
        const uint4 w = *reinterpret_cast<const uint4*>(rc);
        const float2 a0 = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
        const float2 b0 = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
        const float2 a1 = __half22float2(*reinterpret_cast<const __half2*>(&w.z));
        const float2 b1 = __half22float2(*reinterpret_cast<const __half2*>(&w.w));
        const RefT<V2> r{V2(a0.x, a1.x), V2(a0.y, a1.y), V2(b0.x, b1.x), V2(b0.y, b1.y)};
        const V2 s = ref_sum(c, r);
        d[c] = fma(V2(wt<float>(c)), s, d[c]);
        if (cy(c) != 0 && cz(c) != 0) continue;
        const float sl = ref_sum(c, ref1(rc - 1)), sr = ref_sum(c, ref1(rc + 2));
        const float xl = ref1(rc - 1).vx, xr = ref1(rc + 2).vx;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
          if (cy(q) != cy(c) || cz(q) != cz(c) || cx(q) == 0) continue;
          // e_x = 1: upwind nodes x - 1, x; e_x = -1: x + 1, x + 2
          const V2 t = cx(q) == 1 ? V2(sl, lane0(s)) + V2(xl, lane0(r.vx))
                                  : V2(lane1(s), sr) - V2(lane1(r.vx), xr);
          d[q] = fma(V2(wt<float>(q)), t, d[q]);
        }
      }
    }
    if (first) {
#pragma unroll
      for (int q = 1; q < Q; ++q)
        if (cx(q) == 1)
          set0(d[q], xface_value<REF>(p, q, kl, 0, p.up(q),
                                      p.ref - (cz(q) * plane + cy(q) * pitch + 1), nx));
    }
    if (last) {
#pragma unroll
      for (int q = 1; q < Q; ++q)
        if (cx(q) == -1) {
          const float v = xface_value<REF>(p, q, kr, nr, p.up(q) + nr,
                                           p.ref - (cz(q) * plane + cy(q) * pitch - 1) + nr, -nx);
          if (nr == 0) set0(d[q], v);
          else set1(d[q], v);
        }
    }
    return;
  }
  // Rows on a y or z face: the rules select an address per direction (and
  // node, where e_x != 0), so that all loads can be issued together (see
  // pull_face).  A second node in the padding repeats the first.
  const int n1 = x + 1 < nx ? 1 : 0;
  const Faces fA = faces_of(x, y, z, nx, p.ny(), p.nz(), pitch, plane, fb);
  const Faces fB = faces_of(x + n1, y, z, nx, p.ny(), p.nz(), pitch, plane, fb);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int off = cz(q) * plane + cy(q) * pitch + cx(q);
    const bool bA = (fA.wall & up_faces(q)) != 0, bB = (fB.wall & up_faces(q)) != 0;
    const __half *same = p.own(q), *anti = p.own(opp(q));
    const int jA = bA ? 0 : up_wrap(fA, q) - off;
    const int jB = cx(q) == 0 ? jA + n1 : bB ? n1 : up_wrap(fB, q) - off + n1;
    V2 v;
    if (cx(q) == 0) v = ld2((bA ? anti : same) + jA);
    else v = V2(ld1((bA ? anti : same) + jA), ld1((bB ? anti : same) + jB));
    if (REF) {
      // a bounced value is decoded as opp(q): e_q . v changes sign
      const V2 sgn(bA ? -1.0f : 1.0f, bB ? -1.0f : 1.0f);
      const RefT<float> rA = ref1(p.ref + jA), rB = ref1(p.ref + jB);
      const RefT<V2> r{V2(rA.dr, rB.dr), mulr(sgn, V2(rA.vx, rB.vx)), mulr(sgn, V2(rA.vy, rB.vy)),
                       mulr(sgn, V2(rA.vz, rB.vz))};
      v = fma(V2(wt<float>(q)), ref_sum(q, r), v);
    }
    if (fA.lid & up_faces(q)) set0(v, lane0(v) + p.lid(q));
    if (fB.lid & up_faces(q)) set1(v, lane1(v) + p.lid(q));
    d[q] = v;
  }
}

// ---- store ---------------------------------------------------------------
// How a pair's populations are rounded and stored.
enum { PAIR_RN = 0, PAIR_SR = 1, PAIR_REF = 2 };

// The FP16 pair of direction q, stored with one 32-bit access.
__device__ __forceinline__ void st2(__half* p, __half2 v) { *reinterpret_cast<__half2*>(p) = v; }

// The reference of the pair's nodes from density rho = rho0 + drho and
// velocity u: rounded to FP16, stored by one 128-bit access; r receives the
// rounded values.
__device__ __forceinline__ void ref_store2(uint2* p, const NodeOut<V2>& o, float rho0, float lam,
                                           RefT<V2>& r) {
  const V2 r3 = mulr(V2(3.0f * lam), o.rho);
  const V2 dr = mulr(V2(lam), o.rho - V2(rho0));
  const V2 vx = mulr(r3, o.ux), vy = mulr(r3, o.uy), vz = mulr(r3, o.uz);
  const __half2 a0 = __floats2half2_rn(lane0(dr), lane0(vx)),
                b0 = __floats2half2_rn(lane0(vy), lane0(vz)),
                a1 = __floats2half2_rn(lane1(dr), lane1(vx)),
                b1 = __floats2half2_rn(lane1(vy), lane1(vz));
  uint4 w;
  w.x = *reinterpret_cast<const unsigned*>(&a0);
  w.y = *reinterpret_cast<const unsigned*>(&b0);
  w.z = *reinterpret_cast<const unsigned*>(&a1);
  w.w = *reinterpret_cast<const unsigned*>(&b1);
  *reinterpret_cast<uint4*>(p) = w;
  const float2 fa0 = __half22float2(a0), fb0 = __half22float2(b0), fa1 = __half22float2(a1),
               fb1 = __half22float2(b1);
  r = {V2(fa0.x, fa1.x), V2(fa0.y, fa1.y), V2(fb0.x, fb1.x), V2(fb0.y, fb1.y)};
}

// Blocks of 256 threads per SM the pair kernels are compiled for: at most 80
// registers a thread, which all but the forced F16R kernels (one correction
// per population: all 19 inputs live to the end) hold without spills in the
// steps between checks; those take up to 128.
constexpr int pair_min_blocks(bool ref, bool force) { return ref && force ? 2 : 3; }

// Collide the pair.  F16R with a body force takes one correction per
// population (see step_f16r.cu).
template <bool REF, bool FORCE>
__device__ __forceinline__ void collide_pair(const CollideConst<float>& C, V2 (&d)[Q],
                                             NodeOut<V2>& o) {
  collide<V2, FORCE, !REF || !FORCE, log2_scale<__half>(), true>(C, d, o);
}

// Store the pair: dst(q) is its slot of direction q, rdst its reference slot
// (PAIR_REF), i the index of its first node, step the lattice's steps done
// before this one (the random bits depend on these two and the direction
// only, so a lattice alone and in a batch rounds alike).
template <int FORM, typename Dst>
__device__ __forceinline__ void store_pair(const CollideConst<float>& C, V2 (&d)[Q],
                                           const NodeOut<V2>& o, Dst&& dst, uint2* rdst, int i,
                                           unsigned step) {
  if constexpr (FORM == PAIR_RN) {
#pragma unroll
    for (int q = 0; q < Q; ++q) st2(dst(q), __float22half2_rn(d[q].v));
  } else {
    if constexpr (FORM == PAIR_REF) {
      RefT<V2> r;
      ref_store2(rdst, o, C.rho0, float(1 << log2_scale<__half>()), r);
#pragma unroll
      for (int q = 0; q < Q; ++q) d[q] = fma(V2(-wt<float>(q)), ref_sum(q, r), d[q]);
    }
    uint32_t state = sr_seed(uint32_t(i), step);
#pragma unroll
    for (int q = 0; q < Q; ++q)
      *reinterpret_cast<uint32_t*>(dst(q)) = enc16_sr2(lane0(d[q]), lane1(d[q]), state);
  }
}

// The pair's part of the check-step sums; n1: the second node exists.
__device__ __forceinline__ void check_pair(CheckSums& s, const NodeOut<V2>& o, float rho0,
                                           float* up, int64_t nst, bool n1) {
  check_node(s, lane0(o.rho), lane0(o.ux), lane0(o.uy), lane0(o.uz), rho0, up, nst);
  if (n1) check_node(s, lane1(o.rho), lane1(o.ux), lane1(o.uy), lane1(o.uz), rho0, up + 1, nst);
}

// F16R: reference buffers of a lone step; step: the lattice's steps done
// before this one.
struct PairExtra {
  const uint2* ref_src;
  uint2* ref_dst;
  unsigned step;
};

// One time step of a lone lattice; the block is pair_width() threads along x.
template <int FORM, bool FORCE, bool CHECK>
__global__ void __launch_bounds__(256, pair_min_blocks(FORM == PAIR_REF, FORCE))
    step_pair_kernel(const StepArgs<__half, float> a, const PairExtra e) {
  pdl_enter();
  const int x = 2 * int(blockIdx.x * blockDim.x + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = a.zrev ? a.nz - 1 - int(blockIdx.z) : int(blockIdx.z);
  const bool active = x < a.nx && y < a.ny;
  if (!CHECK && !active) return;
  CheckSums sums;
  if (active) {
    const int i = z * a.plane + y * a.pitch + x;
    V2 d[Q];
    NodeOut<V2> o;
    const LonePair p{a, FORM == PAIR_REF ? e.ref_src + i : nullptr, i};
    pull_pair<FORM == PAIR_REF>(p, x, y, z, d);
    collide_pair<FORM == PAIR_REF, FORCE>(a.C, d, o);
    store_pair<FORM>(a.C, d, o, [&](int q) { return a.dstq[q] + i; },
                     FORM == PAIR_REF ? e.ref_dst + i : nullptr, i, e.step);
    if (CHECK)
      check_pair(sums, o, a.C.rho0, static_cast<float*>(a.cb.uprev) + i, int64_t(a.plane) * a.nz,
                 x + 1 < a.nx);
  }
  if (CHECK) block_sums(sums, check_row(a.cb), a.cb.flag);
}

template <int FORM>
cudaError_t launch_step_pair(const StepArgs<__half, float>& a, const PairExtra& e, bool force,
                             bool check, dim3 block, cudaStream_t st) {
  const int threads = int(block.x * block.y), w = pair_width(a.nx, threads);
  const dim3 blk(unsigned(w), unsigned(threads / w));
  const dim3 grid((a.nx + 2 * blk.x - 1) / (2 * blk.x), (a.ny + blk.y - 1) / blk.y, a.nz);
  auto kernel =
      force ? (check ? step_pair_kernel<FORM, true, true> : step_pair_kernel<FORM, true, false>)
            : (check ? step_pair_kernel<FORM, false, true> : step_pair_kernel<FORM, false, false>);
  return pdl_launch(kernel, grid, blk, st, a, e);
}

}  // namespace clbm
