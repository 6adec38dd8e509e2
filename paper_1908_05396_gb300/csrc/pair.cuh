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
// and 49.8 -> 38.6 on 128^3 (224, 5.7 TB/s, and 30 with the face rules as address
// selects); F16R 753 -> 340 and 95 -> 47, whose 19 reference loads a node
// become 9.5 and whose reference is taken off the moments instead of 19
// populations.  DRAM latency and the drain between dependent steps bound F16S
// now; F16R still issues 564 instructions a node (ncu, 128^3: issue 59 % active
// with 23 % of the warps its registers leave).
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
// (dr, v) of a node (RefT), stored as four FP16 values.
__device__ __forceinline__ RefT<float> ref_dec(uint2 v) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
  return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ RefT<float> ref1(const uint2* p) { return ref_dec(*p); }
// dr + e_q . v, the part of the reference term that ref_wt(q) multiplies; the sums
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

// The pre-collision deviations of the pair (x, x + 1) in a row off the y and
// z faces.  XF: some pair of the warp holds x = 0 or x = nx - 1; the nodes
// there take the directions from outside by the face rules of pull_face, each
// by a select of the address (values and references), in the same round of
// loads.
template <bool REF, bool XF, typename P>
__device__ __forceinline__ void pull_row(const P& p, int x, V2 (&d)[Q]) {
  const int nx = p.nx(), pitch = p.pitch(), plane = p.plane();
  const unsigned fb = p.faces();
  const int kl = int(fb & 3u), kr = int((fb >> 2) & 3u);
  // the pair's first node is at x = 0 (fl); its first (f0) or second (f1) node at x = nx - 1
  const bool fl = XF && x == 0, f0 = XF && x + 1 == nx, f1 = XF && x + 2 == nx;
  const bool bl = fl && kl != BC_PERIODIC, b0 = f0 && kr != BC_PERIODIC,
             b1 = f1 && kr != BC_PERIODIC;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const __half* u = p.up(q);
    if (cx(q) == 0) {
      d[q] = ld2(u);
      continue;
    }
    const __half *u0 = u, *u1 = u + 1;
    if (XF) {
      const __half* own = p.own(opp(q));
      if (cx(q) == 1) {
        if (fl) u0 += nx;  // the periodic wrap
        if (bl) u0 = own;  // halfway bounce-back
      } else {
        if (f0) u0 -= nx;
        if (b0) u0 = own;
        if (f1) u1 -= nx;
        if (b1) u1 = own + 1;
      }
    }
    d[q] = V2(ld1(u0), ld1(u1));
  }
  if (REF) {
    // Columns of upwind nodes (e_y, e_z), each one 128-bit reference load for
    // the pair's own x and, where the column's directions have e_x != 0, a
    // 64-bit load on either side.  A bounced value is decoded with the node's
    // own reference as opp(q): e_q . v changes sign.
    const float gl = bl ? -1.0f : 1.0f, g0 = b0 ? -1.0f : 1.0f, g1 = b1 ? -1.0f : 1.0f;
#pragma unroll
    for (int c = 0; c < Q; ++c) {
      if (cx(c) != 0) continue;
      const uint2* rc = p.ref - (cz(c) * plane + cy(c) * pitch);
      const uint4 w = *reinterpret_cast<const uint4*>(rc);
      const RefT<float> a = ref_dec(make_uint2(w.x, w.y)), b = ref_dec(make_uint2(w.z, w.w));
      const RefT<V2> r{V2(a.dr, b.dr), V2(a.vx, b.vx), V2(a.vy, b.vy), V2(a.vz, b.vz)};
      const V2 s = ref_sum(c, r);
      d[c] = fma(V2(ref_wt(c)), s, d[c]);
      if (cy(c) != 0 && cz(c) != 0) continue;
      // left (x - 1) and right (x + 2, and where the pair's first node is the
      // last of the row, x + 1) neighbours, or what stands in for them
      const uint2 *rl = rc - 1, *rr = rc + 2;
      if (XF) {
        if (fl) rl = bl ? p.ref : rl + nx;
        if (f1) rr = b1 ? p.ref + 1 : rr - nx;
        if (f0) rr = b0 ? p.ref : rc + 1 - nx;
      }
      RefT<float> l = ref1(rl), n = ref1(rr);
      float s1 = lane1(s), x1 = lane1(r.vx);
      if (XF) {
        const float gr = g0 * g1;  // (at most one of the two is -1)
        l = {l.dr, mulr(gl, l.vx), mulr(gl, l.vy), mulr(gl, l.vz)};
        n = {n.dr, mulr(gr, n.vx), mulr(gr, n.vy), mulr(gr, n.vz)};
      }
      const float sl = ref_sum(c, l), sn = ref_sum(c, n);
      if (XF && f0) {  // the first node's e_x = -1 value comes from `n`
        s1 = sn;
        x1 = n.vx;
      }
#pragma unroll
      for (int q = 1; q < Q; ++q) {
        if (cy(q) != cy(c) || cz(q) != cz(c) || cx(q) == 0) continue;
        // e_x = 1: upwind nodes x - 1, x; e_x = -1: x + 1, x + 2
        const V2 t = cx(q) == 1 ? V2(sl, lane0(s)) + V2(l.vx, lane0(r.vx))
                                : V2(s1, sn) - V2(x1, n.vx);
        d[q] = fma(V2(ref_wt(q)), t, d[q]);
      }
    }
  }
  if (XF && ((fl && kl == BC_LID) || ((f0 || f1) && kr == BC_LID))) {
#pragma unroll
    for (int q = 1; q < Q; ++q) {
      if (cx(q) == 1 && fl && kl == BC_LID) set0(d[q], lane0(d[q]) + p.lid(q));
      if (cx(q) == -1 && f0 && kr == BC_LID) set0(d[q], lane0(d[q]) + p.lid(q));
      if (cx(q) == -1 && f1 && kr == BC_LID) set1(d[q], lane1(d[q]) + p.lid(q));
    }
  }
}

// F16S: replace the directions that cross an x face after the direct loads.  A
// second round of loads in the threads at x = 0 and x = nx - 1, yet cheaper
// than selecting addresses in all of the warp's (128^3: 30.0 us a step against
// 31.7); F16R, whose patch would load and decode references again, is faster
// the other way (61 and 49 us).
template <typename P>
__device__ __forceinline__ void xface_patch(const P& p, int x, V2 (&d)[Q]) {
  const int nx = p.nx();
  const int kl = int(p.faces() & 3u), kr = int((p.faces() >> 2) & 3u);
  if (x == 0) {
#pragma unroll
    for (int q = 1; q < Q; ++q) {
      if (cx(q) != 1) continue;
      const float v = ld1(kl == BC_PERIODIC ? p.up(q) + nx : p.own(opp(q)));
      set0(d[q], kl == BC_LID ? v + p.lid(q) : v);
    }
  }
  if (x + 2 >= nx) {
    const int n = nx - 1 - x;  // which node of the pair is at nx - 1
#pragma unroll
    for (int q = 1; q < Q; ++q) {
      if (cx(q) != -1) continue;
      float v = ld1(kr == BC_PERIODIC ? p.up(q) + n - nx : p.own(opp(q)) + n);
      if (kr == BC_LID) v += p.lid(q);
      if (n == 0) set0(d[q], v);
      else set1(d[q], v);
    }
  }
}

// The pre-collision deviations of the pair (x, x + 1) in row (y, z).  When nx
// is odd the last pair's second node lies in the row's padding: it is computed
// from whatever is there and stored there.
template <bool REF, typename P>
__device__ __forceinline__ void pull_pair(const P& p, int x, int y, int z, V2 (&d)[Q]) {
  const int nx = p.nx(), pitch = p.pitch(), plane = p.plane();
  const unsigned fb = p.faces();
  if (y > 0 && y < p.ny() - 1 && z > 0 && z < p.nz() - 1) {
    if constexpr (REF) {
      if (__any_sync(__activemask(), x == 0 || x + 2 >= nx)) pull_row<true, true>(p, x, d);
      else pull_row<true, false>(p, x, d);
    } else {
      pull_row<false, false>(p, x, d);
      xface_patch(p, x, d);
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
      v = fma(V2(ref_wt(q)), ref_sum(q, r), v);
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
// velocity u: rounded to FP16 and stored by one 128-bit access; returns the
// rounded values.
__device__ __forceinline__ RefT<V2> ref_store2(uint2* p, const NodeOut<V2>& o, float rho0,
                                               float lam) {
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
  return {V2(fa0.x, fa1.x), V2(fa0.y, fa1.y), V2(fb0.x, fb1.x), V2(fb0.y, fb1.y)};
}

// Blocks of 256 threads per SM the pair kernels are compiled for: up to 80
// registers a thread, for F16R up to 128, which it needs to hold a column's
// references without spills (256^3: 340 us a step, against 352 with 80 and 373
// with 64 registers; F16S with 64 ran at 227 against 224 us there and 31.5
// against 30.0 on 128^3, its stochastic form 243 against 237).
constexpr int pair_min_blocks(bool ref) { return ref ? 2 : 3; }

// Collide the pair and leave in d what is stored: the deviations, or (REF) the
// remainders after the reference, which goes to rdst.  F16R with a body force
// takes one correction per population (see step_f16r.cu).
template <bool REF, bool FORCE>
__device__ __forceinline__ void collide_pair(const CollideConst<float>& C, V2 (&d)[Q],
                                             NodeOut<V2>& o, uint2* rdst) {
  constexpr int L = log2_scale<__half>();
  constexpr float LAM = float(1 << L);
  if constexpr (!REF) {
    collide_unit<V2, FORCE, true, L>(C, d, o);
  } else if constexpr (FORCE) {
    collide_unit<V2, true, false, L>(C, d, o);
    const RefT<V2> r = ref_store2(rdst, o, C.rho0, LAM);
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = fma(V2(-ref_wt(q)), ref_sum(q, r), d[q]);
  } else {
    collide_unit<V2, false, true, L>(
        C, d, o, [&](const NodeOut<V2>& n) { return ref_store2(rdst, n, C.rho0, LAM); });
  }
}

// Store the pair: dst(q) is its slot of direction q, i the index of its first
// node, step the lattice's steps done before this one (the random bits depend
// on these two and the direction only, so a lattice alone and in a batch
// rounds alike); sr: stochastic rounding.
template <typename Dst>
__device__ __forceinline__ void store_pair(const V2 (&d)[Q], bool sr, Dst&& dst, int i,
                                           unsigned step) {
  if (!sr) {
#pragma unroll
    for (int q = 0; q < Q; ++q) st2(dst(q), __float22half2_rn(d[q].v));
    return;
  }
  uint32_t state = sr_seed(uint32_t(i), step);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    *reinterpret_cast<uint32_t*>(dst(q)) = enc16_sr2(lane0(d[q]), lane1(d[q]), state);
}

// The pair's part of the check-step sums; n1: the second node exists.
__device__ __forceinline__ void check_pair(CheckSums& s, const NodeOut<V2>& o, float rho0,
                                           float* up, int64_t nst, bool n1) {
  check_node(s, lane0(o.rho), lane0(o.ux), lane0(o.uy), lane0(o.uz), rho0, up, nst);
  if (n1) check_node(s, lane1(o.rho), lane1(o.ux), lane1(o.uy), lane1(o.uz), rho0, up + 1, nst);
}

// F16R: reference buffers of a lone step; seed: the lattice's steps done
// before this one.
struct PairExtra {
  const uint2* ref_src;
  uint2* ref_dst;
  StepSeed seed;
};

// One time step of a lone lattice; the block is pair_width() threads along x.
template <int FORM, bool FORCE, bool CHECK>
__global__ void __launch_bounds__(256, pair_min_blocks(FORM == PAIR_REF))
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
    collide_pair<FORM == PAIR_REF, FORCE>(a.C, d, o, e.ref_dst + i);
    store_pair(d, FORM != PAIR_RN, [&](int q) { return a.dstq[q] + i; }, i,
               FORM != PAIR_RN ? e.seed.get() : 0u);
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
