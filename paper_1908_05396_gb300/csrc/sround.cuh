// sround.cuh -- stochastically rounded FP16 stores, shared by the step
// kernels that use them (the F16R form, and the F16S form with stochastic
// rounding).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace clbm {

// The lattice's step count that seeds a step's rounding: a constant of the
// launch, or relative to a count in device memory (a launch in a graph that
// is replayed).
struct StepSeed {
  unsigned step = 0;
  const unsigned* base = nullptr;
  __device__ __forceinline__ unsigned get() const { return base ? *base + step : step; }
};

// Stochastic rounding of the stores: a value is rounded up in magnitude with
// probability equal to the fraction of an FP16 ulp it carries, so increments
// far below one ulp (a weak body force, a slow transient) survive on average
// instead of being rounded away every step.  The random bits depend only on
// the node index, the direction and the lattice's own step count, so a
// lattice gives the same result alone and in a batch, and stepped one or two
// nodes per thread: one integer hash of (node pair, step) (the finaliser of
// MurmurHash3), then one step per direction of a 32-bit linear congruential
// generator with the multiplier and increment of PCG (O'Neill, 2014), whose
// word rounds the direction's two values of the nodes 2k and 2k + 1.
__device__ __forceinline__ uint32_t sr_seed(uint32_t node, uint32_t step) {
  uint32_t h = (node & ~1u) ^ (step * 0x9E3779B9u);
  h ^= h >> 16;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return h;
}

// The values of an even node and the odd one after it at once, with the
// GB300's stochastic-rounding conversion (cvt.rs.f16x2.f32: each value rounded
// up in magnitude with the probability of the fraction of an FP16 ulp it
// carries), packed in memory order (the even node in the lower half).  The
// conversion adds the low 13 bits of each 16-bit half of the random word
// below the kept mantissa (measured: bits 0-12 round the lower value, bits
// 16-28 the upper).  The generator's upper half is folded into the lower one:
// the low bits of a power-of-two-modulus LCG have short periods, its high
// bits do not.
__device__ __forceinline__ uint32_t enc16_sr2(float even, float odd, uint32_t& state) {
  state = state * 747796405u + 2891336453u;
  const uint32_t rbits = state ^ (state >> 16);
  uint32_t d;
  asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;"
      : "=r"(d)
      : "f"(odd), "f"(even), "r"(rbits));
  return d;
}

// The value of one node (odd: bit 0 of its index), rounded as in its pair.
__device__ __forceinline__ __half enc16_sr1(float v, uint32_t odd, uint32_t& state) {
  return __ushort_as_half(static_cast<unsigned short>(enc16_sr2(v, v, state) >> (16 * odd)));
}

// The 19 values of node i (index in its lattice) after `step` earlier steps.
template <typename Dst, int N>
__device__ __forceinline__ void store_sr1(Dst&& dst, const float (&d)[N], uint32_t i,
                                          uint32_t step) {
  uint32_t state = sr_seed(i, step);
#pragma unroll
  for (int q = 0; q < N; ++q) *dst(q) = enc16_sr1(d[q], i & 1u, state);
}

}  // namespace clbm
