// batch.cuh -- one persistent launch that steps many lattices of uneven size.
//
// Every lattice is cut into tiles of (block_x x block_y) nodes of one plane.
// A device table maps each tile to its lattice, and each lattice has a
// descriptor (buffers, geometry, collision constants) in a __constant__ table
// of the translation unit.  A persistent grid of blocks strides over the
// tiles.  Lattices with a body force come last in the tile table and are
// stepped by a second launch compiled with the force path, so neither kernel
// carries the registers of both paths.  Parameters live in device memory, so
// a CUDA graph captured once stays valid when lattices join or leave: only
// the tables change.
#pragma once

#include "kernels.cuh"
#include "sround.cuh"

namespace clbm {

template <typename R>
struct LatDesc {
  const void* buf[2];  // buf[p]: source buffer at parity p (the other is the destination)
  const void* ref[2];  // F16R form: the reference moments kept with buf[p] (else null)
  void* uprev;         // velocities of the previous check (math type)
  int64_t qstride;
  int nx, ny, nz, pitch, plane;
  unsigned facebits;
  int tiles_x, tiles_y;
  int tw_log2;         // tile width (nodes along x) = 1 << tw_log2, height = threads / width
  int slot;            // row of this lattice in the batch's reduction array
  unsigned step_offset;  // lattice steps minus batch steps (seeds stochastic rounding)
  int sround;            // F16S: stores rounded stochastically
  int threads;           // threads per block the tiles were cut for; 0: not usable
  R lidc[Q];
  CollideConst<R> C;
};

// One node of the batched step: same pull, boundaries and collision as
// step_kernel.  Source offsets are formed from compile-time direction
// constants right before each load, so no per-direction table is held in
// registers.
template <typename S, typename R, bool FORCE, bool UNIT>
__device__ __forceinline__ void batch_node(const LatDesc<R>& L, const S* __restrict__ src,
                                           S* __restrict__ dst, int x, int y, int z,
                                           unsigned step, NodeOut<R>& o) {
  const int qs = int(L.qstride), plane = L.plane, pitch = L.pitch;
  const int i = z * plane + y * pitch + x;
  R d[Q];
  // as pull_node: warps off every face load directly
  const bool inner = y > 0 && y < L.ny - 1 && z > 0 && z < L.nz - 1 && x > 0 && x < L.nx - 1;
  if (__all_sync(__activemask(), inner)) {
#pragma unroll
    for (int q = 0; q < Q; ++q)
      d[q] = Codec<S, R>::dec(src[q * qs + i - (cz(q) * plane + cy(q) * pitch + cx(q))], R(1));
  } else {
    pull_face<S, R>(src, L.qstride, L.nx, L.ny, L.nz, pitch, plane, L.facebits, x, y, z, i,
                    L.lidc, d);
  }
  collide<R, FORCE, pair_out<S>(), log2_scale<S>(), UNIT>(L.C, d, o);
  if constexpr (std::is_same<S, __half>::value) {
    if (L.sround) {
      store_sr1([&](int q) { return dst + (q * qs + i); }, d, uint32_t(i), step);
      return;
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) dst[q * qs + i] = Codec<S, R>::enc(d[q], R(1));
}

// One node of the batched step in the F16R form, any rates (defined with the
// other F16R kernels, the only translation unit that instantiates the batch
// with REF).
template <bool FORCE>
__device__ void batch_node_ref(const LatDesc<float>& L, int parity, int x, int y, int z,
                               unsigned step, NodeOut<float>& o);

// A pair's upwind values in a lattice of the batch (see LonePair).
struct BatchPair {
  const LatDesc<float>& L;
  const __half* src;  // the pair's own value of direction 0
  const uint2* ref;
  int qs;
  __device__ __forceinline__ const __half* up(int q) const {
    return src + (q * qs - (cz(q) * L.plane + cy(q) * L.pitch + cx(q)));
  }
  __device__ __forceinline__ const __half* own(int q) const { return src + q * qs; }
  __device__ __forceinline__ int nx() const { return L.nx; }
  __device__ __forceinline__ int ny() const { return L.ny; }
  __device__ __forceinline__ int nz() const { return L.nz; }
  __device__ __forceinline__ int pitch() const { return L.pitch; }
  __device__ __forceinline__ int plane() const { return L.plane; }
  __device__ __forceinline__ unsigned faces() const { return L.facebits; }
  __device__ __forceinline__ float lid(int q) const { return L.lidc[q]; }
};

// Two nodes along x of the batched step of an FP16 form: the pull, collision
// and store of step_pair_kernel.
template <bool FORCE, bool REF>
__device__ __forceinline__ void batch_pair(const LatDesc<float>& L, int parity, int x, int y, int z,
                                           unsigned step, NodeOut<V2>& o) {
  const int i = z * L.plane + y * L.pitch + x, qs = int(L.qstride);
  const __half* src = static_cast<const __half*>(L.buf[parity]) + i;
  __half* out = static_cast<__half*>(const_cast<void*>(L.buf[parity ^ 1])) + i;
  const uint2* rs = REF ? static_cast<const uint2*>(L.ref[parity]) + i : nullptr;
  uint2* rd = REF ? static_cast<uint2*>(const_cast<void*>(L.ref[parity ^ 1])) + i : nullptr;
  V2 d[Q];
  pull_pair<REF>(BatchPair{L, src, rs, qs}, x, y, z, d);
  collide_pair<REF, FORCE>(L.C, d, o, rd);
  store_pair(d, REF || L.sround != 0, [&](int q) { return out + q * qs; }, i, step);
}

// tile word: x tile (8 bits) | y tile (12 bits) | z chunk (12 bits)
__host__ __device__ __forceinline__ unsigned tile_word(int tx, int ty, int tz) {
  return unsigned(tx) | (unsigned(ty) << 8) | (unsigned(tz) << 20);
}

// The tile loop of the batched step.  get(li) returns lattice li's
// descriptor from the translation unit's __constant__ table, so ptxas can
// reload its fields where it needs them instead of holding them in registers.
template <typename S, typename R, bool CHECK, bool FORCE, bool REF, bool UNIT, typename Get>
__device__ __forceinline__ void batch_tiles(Get get, const int* __restrict__ owner,
                                            const unsigned* __restrict__ coord,
                                            BatchHeader* hdr, int parity, double* acc, int zc) {
  // F16R and F16S (whose lattices may round stochastically): this group's
  // step count, advanced at the end of each of its launches by the launch's
  // last CTA
  constexpr bool PAIR = UNIT && std::is_same<S, __half>::value;
  constexpr int GROUP = (FORCE ? 2 : 0) + (UNIT ? 0 : 1);
  constexpr bool STEPS = REF || std::is_same<S, __half>::value;
  const unsigned bstep =
      STEPS ? *reinterpret_cast<volatile const unsigned*>(&hdr->step[GROUP]) : 0u;
  const int t0 = GROUP ? hdr->tile_end[GROUP ? GROUP - 1 : 0] : 0;
  const int t1 = hdr->tile_end[GROUP];
  const int nlat = hdr->nlat;
  // The next tile's table entries are loaded while this tile collides, so a
  // tile starts with one dependent round trip (descriptor) instead of two.
  int t = t0 + int(blockIdx.x);
  int li_next = t < t1 ? owner[t] : 0;
  unsigned w_next = t < t1 ? coord[t] : 0u;
  for (; t < t1; t += gridDim.x) {
    const int li = li_next;
    const unsigned w = w_next;
    if (t + int(gridDim.x) < t1) {
      li_next = owner[t + gridDim.x];
      w_next = coord[t + gridDim.x];
    }
    const int tx = int(w & 0xffu), ty = int((w >> 8) & 0xfffu), tz = int(w >> 20);
    // Self-check of the tables before any access through them.  What does not
    // depend on the tile was checked when the descriptor was filled
    // (usable_desc), which leaves `threads` 0 otherwise.
    bool ok = li >= 0 && li < nlat;
    const LatDesc<R>& L = get(ok ? li : 0);
    if (ok)
      ok = L.threads == int(blockDim.x * blockDim.y) && tx < L.tiles_x && ty < L.tiles_y &&
           zc >= 1 && tz * zc < L.nz && (L.C.has_force != 0) == FORCE;
    if (!ok) {  // block-uniform: skip the tile, report it
      if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(&hdr->err, 1);
      continue;
    }
    // the block's threads in row order over a tile of 2^tw_log2 x (threads
    // >> tw_log2) nodes, or node pairs (the tile width is chosen per lattice)
    const int lin = int(threadIdx.y * blockDim.x + threadIdx.x);
    const int xt = (tx << L.tw_log2) + (lin & ((1 << L.tw_log2) - 1));
    const int x = PAIR ? 2 * xt : xt;
    const int y = ty * (int(blockDim.x * blockDim.y) >> L.tw_log2) + (lin >> L.tw_log2);
    const S* src = static_cast<const S*>(L.buf[parity]);
    S* dst = static_cast<S*>(const_cast<void*>(L.buf[parity ^ 1]));
    const bool active = x < L.nx && y < L.ny;
    CheckSums sums;
    // the tile's zc planes: the per-tile work (table entries, descriptor,
    // checks, the check-step reductions) is shared by zc nodes per thread
    const int z1 = min(tz * zc + zc, L.nz);
#pragma unroll 1
    for (int z = tz * zc; z < z1; ++z) {
      if (active) {
        if constexpr (PAIR) {
          NodeOut<V2> o;
          batch_pair<FORCE, REF>(L, parity, x, y, z, bstep + L.step_offset, o);
          if (CHECK)
            check_pair(sums, o, L.C.rho0,
                       static_cast<float*>(L.uprev) + (z * L.plane + y * L.pitch + x),
                       int64_t(L.plane) * L.nz, x + 1 < L.nx);
          continue;
        }
        NodeOut<R> o;
        if constexpr (REF) batch_node_ref<FORCE>(L, parity, x, y, z, bstep + L.step_offset, o);
        else batch_node<S, R, FORCE, UNIT>(L, src, dst, x, y, z, bstep + L.step_offset, o);
        if (CHECK)
          check_node(sums, o.rho, o.ux, o.uy, o.uz, L.C.rho0,
                     static_cast<R*>(L.uprev) + (z * L.plane + y * L.pitch + x),
                     int64_t(L.plane) * L.nz);
      }
    }
    if (CHECK) {
      double* a = acc + 4 * BATCH_ROWS * L.slot;
      block_sums(sums, a + 4 * (t & (BATCH_ROWS - 1)), reinterpret_cast<int*>(a + 3));
    }
  }
  if constexpr (STEPS) {
    // every CTA of this launch has read its chain's step count: the last one
    // to finish advances it
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      __threadfence();
      if (atomicAdd(&hdr->done[GROUP], 1) == int(gridDim.x) - 1) {
        atomicExch(&hdr->done[GROUP], 0);
        atomicAdd(&hdr->step[GROUP], 1u);
      }
    }
  }
}

// Blocks of 256 threads per SM that the batch kernel is compiled for: 64
// registers when capped, what it likes when not; kernels that step two nodes
// per thread have one variant (launched for both) with 80, or 128, registers.
template <typename S>
constexpr int batch_min_blocks(bool cap, bool unit, bool ref) {
  return std::is_same<S, __half>::value && unit ? pair_min_blocks(ref) : cap ? 4 : 1;
}

// The grid of a persistent launch: per_sm blocks per SM, but no more than fit
// at once (a block beyond them would start its share of the tiles only when
// another has finished all of its own).
inline int batch_grid(const void* kernel, dim3 block, int per_sm, int sms) {
  int fit = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, int(block.x * block.y), 0) !=
          cudaSuccess || fit < 1)
    return per_sm * sms;
  return (per_sm < fit ? per_sm : fit) * sms;
}

// Bytes of __constant__ memory given to the descriptor table of one storage
// form; batches reserve disjoint ranges of it.
constexpr int BATCH_CONST_BYTES = 60 * 1024;

// Whether a descriptor is consistent, for blocks of `threads` threads.
template <typename R>
bool usable_desc(const LatDesc<R>& L, int threads, bool ref) {
  return L.buf[0] && L.buf[1] && L.tw_log2 >= 0 && L.tw_log2 <= 10 &&
         (1 << L.tw_log2) <= threads && threads % (1 << L.tw_log2) == 0 && L.pitch >= L.nx &&
         L.plane == L.pitch * L.ny && L.qstride >= int64_t(L.plane) * L.nz &&
         19 * L.qstride < (int64_t(1) << 31) && (!ref || (L.ref[0] && L.ref[1]));
}

// Host-side fill of one descriptor (constants converted once, in double).
template <typename R>
void fill_desc_t(void* out, double lam, const Geom& g, const PhysParams& P, const void* cur,
                 const void* other,
                 const void* ref_cur, const void* ref_other, void* uprev, int tiles_x,
                 int tiles_y, int tw_log2, int slot, unsigned step_offset, int threads,
                 bool ref) {
  LatDesc<R> L{};
  L.buf[0] = cur;
  L.buf[1] = other;
  L.ref[0] = ref_cur;
  L.ref[1] = ref_other;
  L.uprev = uprev;
  L.qstride = g.qstride;
  L.nx = g.nx;
  L.ny = g.ny;
  L.nz = g.nz;
  L.pitch = g.pitch;
  L.plane = int(g.plane);
  L.facebits = g.facebits;
  L.tiles_x = tiles_x;
  L.tiles_y = tiles_y;
  L.tw_log2 = tw_log2;
  L.slot = slot;
  L.step_offset = step_offset;
  L.sround = 0;
  for (int q = 0; q < Q; ++q)
    L.lidc[q] = R(6.0 * wt<double>(q) * g.rho0 * lam *
                  (cx(q) * g.U[0] + cy(q) * g.U[1] + cz(q) * g.U[2]));
  L.C = make_const<R>(P, lam);
  L.threads = usable_desc(L, threads, ref) ? threads : 0;
  *static_cast<LatDesc<R>*>(out) = L;
}

}  // namespace clbm

#define CLBM_DEFINE_BATCH(SUFFIX, S, R, REF)                                                   \
  namespace clbm {                                                                             \
  __constant__ LatDesc<R> c_lat_##SUFFIX[BATCH_CONST_BYTES / sizeof(LatDesc<R>)];              \
  template <bool CHECK, bool CAP, bool FORCE, bool UNIT>                                       \
  __global__ void __launch_bounds__(256, batch_min_blocks<S>(CAP, UNIT, REF))                  \
      batch_kernel_##SUFFIX(int base, const int* __restrict__ owner,                           \
                            const unsigned* __restrict__ coord, BatchHeader* hdr, int parity,  \
                            double* acc, int zc) {                                             \
    batch_tiles<S, R, CHECK, FORCE, REF, UNIT>(                                                \
        [base](int li) -> const LatDesc<R>& { return c_lat_##SUFFIX[base + li]; }, owner,      \
        coord, hdr, parity, acc, zc);                                                          \
  }                                                                                            \
  cudaError_t launch_batch_##SUFFIX(int base, const int* owner, const unsigned* coord,         \
                                    const void* hdr, int parity, bool check, double* acc,      \
                                    int zc, dim3 block, int per_sm, bool cap, int sms,         \
                                    bool rates, cudaStream_t st, cudaStream_t stf) {           \
    BatchHeader* H = static_cast<BatchHeader*>(const_cast<void*>(hdr));                        \
    auto go = [&](void (*k)(int, const int*, const unsigned*, BatchHeader*, int, double*, int), \
                  cudaStream_t s) {                                                            \
      k<<<batch_grid(reinterpret_cast<const void*>(k), block, per_sm, sms), block, 0, s>>>(    \
          base, owner, coord, H, parity, acc, zc);                                             \
    };                                                                                         \
    /* tiles without force on st, tiles with force on stf (an empty range exits at once) */   \
    if (std::is_same<S, __half>::value) cap = true;                                            \
    auto k0 = check ? (cap ? batch_kernel_##SUFFIX<true, true, false, true>                    \
                           : batch_kernel_##SUFFIX<true, false, false, true>)                  \
                    : (cap ? batch_kernel_##SUFFIX<false, true, false, true>                   \
                           : batch_kernel_##SUFFIX<false, false, false, true>);                \
    auto k1 = check ? (cap ? batch_kernel_##SUFFIX<true, true, true, true>                     \
                           : batch_kernel_##SUFFIX<true, false, true, true>)                   \
                    : (cap ? batch_kernel_##SUFFIX<false, true, true, true>                    \
                           : batch_kernel_##SUFFIX<false, false, true, true>);                 \
    go(k0, st);                                                                                \
    go(k1, stf);                                                                               \
    if (rates) { /* some lattice has other rates omega_9..18: their tiles */                   \
      go(check ? batch_kernel_##SUFFIX<true, false, false, false>                              \
               : batch_kernel_##SUFFIX<false, false, false, false>, st);                       \
      go(check ? batch_kernel_##SUFFIX<true, false, true, false>                               \
               : batch_kernel_##SUFFIX<false, false, true, false>, stf);                       \
    }                                                                                          \
    return cudaGetLastError();                                                                 \
  }                                                                                            \
  size_t desc_size_##SUFFIX() { return sizeof(LatDesc<R>); }                                    \
  int desc_capacity_##SUFFIX() { return int(BATCH_CONST_BYTES / sizeof(LatDesc<R>)); }         \
  void fill_desc_##SUFFIX(void* out, const Geom& g, const PhysParams& P, const void* cur,        \
                          const void* other, const void* ref_cur, const void* ref_other,       \
                          void* uprev, int tx, int ty, int twl, int slot, unsigned so,         \
                          int threads) {                                                       \
    /* FP16 storage (F16S, F16R) carries its deviations scaled by 1024 */                    \
    fill_desc_t<R>(out, double(1 << log2_scale<S>()), g, P, cur, other, ref_cur,             \
                   ref_other, uprev, tx, ty, twl, slot, so, threads, REF);                     \
  }                                                                                            \
  void desc_set_sround_##SUFFIX(void* out, int on) {                                           \
    static_cast<LatDesc<R>*>(out)->sround = on;                                                \
  }                                                                                            \
  cudaError_t upload_desc_##SUFFIX(const void* host, int base, int n) {                        \
    return cudaMemcpyToSymbol(c_lat_##SUFFIX, host, size_t(n) * sizeof(LatDesc<R>),            \
                              size_t(base) * sizeof(LatDesc<R>), cudaMemcpyHostToDevice);      \
  }                                                                                            \
  }
