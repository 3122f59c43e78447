// philox_noise.cuh -- the noise stream's Philox4x32-10 (Salmon, Moraes, Dror,
// Shaw, SC'11) split into what a voice fixes and what a block changes.
//
// Block q of voice g (samples 4q .. 4q + 3, Sec. 2.1 deterministic noise) is
// Philox4x32-10 of the counter (g lo, g hi, q, stream) under the key (seed lo,
// seed hi). Only the third counter word changes along a voice, so beside the
// key schedule two of the rounds' products are fixed by the voice: round 1
// multiplies counter word 0 (g lo), and round 2 multiplies round 1's third
// word, which is made of g lo, the stream and the key only. philox_noise_setup
// computes those fixed parts once (per tile); philox_noise then takes 55
// integer operations per block instead of the plain rounds' 78 (ten rounds of
// two high and two low products, two three-way xors and two key additions),
// with a bit-identical result.
//
// The fractional-rate audio loop of the fused render uses it (3.5% less time
// per batch at 16 kHz, and that loop no longer spills). The integer-rate loop
// keeps the plain rounds, which measured 1.2% faster there, as did a lighter
// split that holds only the first three rounds' fixed parts. The normalised
// renders, at either rate, read the fixed parts from shared memory
// (philox_noise_shared).
//
// Host-compilable (plain C++ outside nvcc) so that a CPU test can compare it
// with the plain rounds.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define SYNTH_PHILOX_HD __host__ __device__ __forceinline__
#else
#define SYNTH_PHILOX_HD inline
#endif

namespace synth {

constexpr uint32_t kPhiloxM0 = 0xD2511F53u;  // multiplier of counter word 0
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;  // multiplier of counter word 2
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;  // Weyl increments of the key words
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

SYNTH_PHILOX_HD uint32_t philox_mulhi(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * (uint64_t)b) >> 32);
#endif
}

// The parts of the rounds that the fixed counter words and the key determine.
// Round r (r = 1..10) uses key (k0 + (r - 1) W0, k1 + (r - 1) W1).
struct PhiloxNoise {
  uint32_t x1;            // round 1: word 1 ^ key word 0 (xor-ed into high(M1 q))
  uint32_t x2;            // round 2: high(M1 z1) ^ key word 0 (xor-ed into low(M1 q))
  uint32_t z2;            // round 2: low(M0 word 0) ^ key word 1
  uint32_t x3;            // round 3: low(M1 z1) ^ key word 0
  uint32_t z3;            // round 3: key word 1
  uint32_t k[14];         // keys of rounds 4..10 (word 0, word 1 of each)
  uint32_t pad;
};

SYNTH_PHILOX_HD PhiloxNoise philox_noise_setup(uint32_t c0, uint32_t c1, uint32_t c3, uint32_t k0,
                                               uint32_t k1) {
  PhiloxNoise p;
  // round 1: word 0's product and the new third word z1 are fixed
  const uint32_t z1 = philox_mulhi(kPhiloxM0, c0) ^ c3 ^ k1;
  const uint32_t w1 = kPhiloxM0 * c0;
  p.x1 = c1 ^ k0;
  k0 += kPhiloxW0;
  k1 += kPhiloxW1;
  // round 2: the product of z1 is fixed; its low half becomes word 1 of round 3
  p.x2 = philox_mulhi(kPhiloxM1, z1) ^ k0;
  const uint32_t y2 = kPhiloxM1 * z1;
  p.z2 = w1 ^ k1;
  k0 += kPhiloxW0;
  k1 += kPhiloxW1;
  p.x3 = y2 ^ k0;
  p.z3 = k1;
#pragma unroll
  for (int r = 0; r < 7; ++r) {
    k0 += kPhiloxW0;
    k1 += kPhiloxW1;
    p.k[2 * r] = k0;
    p.k[2 * r + 1] = k1;
  }
  p.pad = 0;
  return p;
}

// Philox4x32-10 of the counter (c0, c1, q, c3) under (k0, k1), given
// philox_noise_setup(c0, c1, c3, k0, k1).
SYNTH_PHILOX_HD void philox_noise(const PhiloxNoise& p, uint32_t q, uint32_t out[4]) {
  // round 1: (high(M1 q) ^ c1 ^ k0, low(M1 q), fixed, fixed)
  const uint32_t x1 = philox_mulhi(kPhiloxM1, q) ^ p.x1;
  const uint32_t y1 = kPhiloxM1 * q;
  // round 2: word 0's product varies, word 2's is fixed
  uint32_t x = y1 ^ p.x2;
  uint32_t z = philox_mulhi(kPhiloxM0, x1) ^ p.z2;
  uint32_t w = kPhiloxM0 * x1;
  // round 3: word 1 (low(M1 z1)) is fixed and folded into p.x3
  uint32_t h0 = philox_mulhi(kPhiloxM0, x), l0 = kPhiloxM0 * x;
  uint32_t h1 = philox_mulhi(kPhiloxM1, z), l1 = kPhiloxM1 * z;
  x = h1 ^ p.x3;
  uint32_t y = l1;
  z = h0 ^ w ^ p.z3;
  w = l0;
  // rounds 4..10
#pragma unroll
  for (int r = 0; r < 7; ++r) {
    h0 = philox_mulhi(kPhiloxM0, x);
    l0 = kPhiloxM0 * x;
    h1 = philox_mulhi(kPhiloxM1, z);
    l1 = kPhiloxM1 * z;
    x = h1 ^ y ^ p.k[2 * r];
    y = l1;
    z = h0 ^ w ^ p.k[2 * r + 1];
    w = l0;
  }
  out[0] = x;
  out[1] = y;
  out[2] = z;
  out[3] = w;
}

#if defined(__CUDACC__)
// The same with the fixed parts in shared memory (16-byte aligned), loaded
// where they are used, four words at a time: held in registers, or left to the
// compiler to hoist, they spill the render's audio loop. The loads are marked as
// reading memory, so that no ordinary store to *p may pass them.
__device__ __forceinline__ uint4 philox_noise_shared(const PhiloxNoise* p, uint32_t q) {
  const uint32_t at = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t f[4];
  auto fixed = [&](int i) {
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3])
                 : "r"(at + 16 * i)
                 : "memory");
  };
  auto product = [](uint32_t m, uint32_t a, uint32_t& hi, uint32_t& lo) {
    hi = __umulhi(m, a);
    lo = m * a;
  };
  fixed(0);
  uint32_t h0, l0, h1, l1, x, y, z, w;
  product(kPhiloxM1, q, h1, l1);
  product(kPhiloxM0, h1 ^ f[0], h0, w);
  x = l1 ^ f[1];
  z = h0 ^ f[2];
  product(kPhiloxM0, x, h0, l0);
  product(kPhiloxM1, z, h1, l1);
  x = h1 ^ f[3];
  y = l1;
  fixed(1);
  z = h0 ^ w ^ f[0];
  w = l0;
#pragma unroll
  for (int r = 0; r < 7; ++r) {
    product(kPhiloxM0, x, h0, l0);
    product(kPhiloxM1, z, h1, l1);
    // word 5 + 2 r of the struct, then 6 + 2 r
    x = h1 ^ y ^ f[(1 + 2 * r) & 3];
    y = l1;
    if ((2 + 2 * r) % 4 == 0) fixed(1 + (2 + 2 * r) / 4);
    z = h0 ^ w ^ f[(2 + 2 * r) & 3];
    w = l0;
  }
  return make_uint4(x, y, z, w);
}
#endif

}  // namespace synth
