// Device-side random numbers of the NetMax round simulator: Philox4x32-10 (Salmon, Moraes,
// Dror, Shaw, SC'11) and a Box-Muller transform on fixed-point uniforms.
//
// The paper only assumes additive gradient noise with zero mean and bounded variance
// (Assumption 1); the generator, the counter layout and the uniform-to-normal map are this
// library's choice and are documented in the C header's conventions.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace netmax {

constexpr uint32_t kPhiloxMul0 = 0xD2511F53u;
constexpr uint32_t kPhiloxMul1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxWeyl0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxWeyl1 = 0xBB67AE85u;

// Streams (fourth counter word, low byte).
constexpr uint32_t kTagPeer = 1, kTagNoise = 2, kTagX0 = 3, kTagC = 4;

// The ten round keys of one seed, expanded once on the host (the key schedule does not
// depend on the counter, so every thread shares it).
struct PhiloxKeys {
  uint32_t k0[10];
  uint32_t k1[10];
};

inline PhiloxKeys make_philox_keys(uint64_t seed) {
  PhiloxKeys k;
  uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    k.k0[r] = a;
    k.k1[r] = b;
    a += kPhiloxWeyl0;
    b += kPhiloxWeyl1;
  }
  return k;
}

// Counter layout: (column group e/4, worker, round low word, tag | round high bits << 8).
__host__ __device__ __forceinline__ uint32_t philox_ctr3(uint32_t tag, uint64_t round) {
  return tag | ((uint32_t)(round >> 32) << 8);
}

__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               const PhiloxKeys& keys) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)kPhiloxMul0 * c0;  // one 32x32->64 multiply each
    const uint64_t p1 = (uint64_t)kPhiloxMul1 * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ keys.k0[r];
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ keys.k1[r];
    c0 = n0;
    c1 = (uint32_t)p1;
    c2 = n2;
    c3 = (uint32_t)p0;
  }
  return make_uint4(c0, c1, c2, c3);
}

// How the same operations, with the same results, are issued.  Which form is faster is each kernel's own (its registers,
// what else it issues), so every kernel names its form beside the figures.
constexpr int kPairs = 1;   // the step along the gradient on fp32 pairs, not as scalars
constexpr int kFunnel = 2;  // the radius's mantissa by one funnel shift instead of a shift and an or

// u1 = (top23(a) + 1/2) / 2^23 in (0,1), exactly representable in fp32:
// bits 0x3F800000 | top23 are the float 1 + top23 / 2^23; subtracting 1 - 2^-24 is exact.
template <int kForm = 0>
__device__ __forceinline__ float radius_uniform(uint32_t a) {
  if (!(kForm & kFunnel)) return __uint_as_float(0x3F800000u | (a >> 9)) - 0.99999994039535522461f;
  // (those bits are the funnel shift of 0x7F : a by 9)
  return __uint_as_float(__funnelshift_r(a, 0x7Fu, 9)) - 0.99999994039535522461f;
}

// Hardware log2 of a normal number (u1 >= 2^-24 here, so flushing subnormals changes nothing
// and saves the subnormal-input handling around the instruction).
__device__ __forceinline__ float log2_fast(float v) {
#ifdef NETMAX_LG2_NO_FTZ
  return __log2f(v);
#else
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
#endif
}

// Accurate pair (library logf / sincospif / sqrtf): used where speed does not matter.
__device__ __forceinline__ void normal_pair_accurate(uint32_t a, uint32_t b, float& z0, float& z1) {
  const float u1 = radius_uniform(a);
  const float turns2 = (float)((int32_t)b >> 8) * 1.1920928955078125e-07f;  // 2 u2 in [-1, 1)
  const float rad = sqrtf(-2.0f * logf(u1));
  float s, c;
  sincospif(turns2, &s, &c);
  z0 = rad * c;
  z1 = rad * s;
}

// ---- packed fp32x2 arithmetic (sm_100: two IEEE fp32 operations per instruction) ----------
typedef unsigned long long pair_t;  // two floats in one 64-bit register: (low lane, high lane)

__device__ __forceinline__ pair_t pack2(float lo, float hi) {
  pair_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(pair_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c) {
  pair_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ pair_t add2(pair_t a, pair_t b) {
  pair_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// sub.rn.f32x2 is a - b in each lane.
__device__ __forceinline__ pair_t sub2(pair_t a, pair_t b) {
  pair_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// A Box-Muller pair times sigma, fast path: (sigma_s rad) (cos, sin) of 2 pi u2 with rad = sqrt(-log2 u1);
// sigma_s is sigma times the constant factor kNormalScale = sqrt(2 ln 2) that rad leaves out.
// u1 < 1, so log2 u1 < 0; the hardware logarithm has an absolute error of about 2^-22 and may
// return +0 or a tiny positive value for u1 next to 1, hence |.| (an operand modifier, not an
// instruction) instead of a negation under the square root.
constexpr double kNormalScale = 1.17741002251547469101;  // sqrt(2 ln 2)
template <int kForm>
__device__ __forceinline__ pair_t scaled_pair(uint32_t a, uint32_t b, float sigma_s) {
  const float u1 = radius_uniform<kForm>(a);
  const float ang = (float)((int32_t)b >> 8) * 3.74507028e-07f;  // 2 pi / 2^24
  float rad;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rad) : "f"(fabsf(log2_fast(u1))));
  rad *= sigma_s;
  float s, c;
  __sincosf(ang, &s, &c);
  return pack2(rad * c, rad * s);  // (not on pairs: the compiler contracts a packed product with the sum that follows, other bits)
}
// sigma times the four normals of a Philox block.
template <int kForm>
__device__ __forceinline__ ulonglong2 scaled_normals4(uint4 r, float sigma_s) {
  return make_ulonglong2(scaled_pair<kForm>(r.x, r.y, sigma_s), scaled_pair<kForm>(r.z, r.w, sigma_s));
}
// Clears the lanes from `live` on (padding of a row's last, ragged group).
__device__ __forceinline__ ulonglong2 mask_lanes(ulonglong2 v, int live) {
  float v0, v1, v2, v3;
  unpack2(v.x, v0, v1);
  unpack2(v.y, v2, v3);
  return make_ulonglong2(pack2(live > 0 ? v0 : 0.f, live > 1 ? v1 : 0.f), pack2(live > 2 ? v2 : 0.f, live > 3 ? v3 : 0.f));
}

// The four normals of a Philox block, accurate (initial state).
__device__ __forceinline__ float4 normals4(uint4 r) {
  float4 z;
  normal_pair_accurate(r.x, r.y, z.x, z.y);
  normal_pair_accurate(r.z, r.w, z.z, z.w);
  return z;
}

// ---- noise blocks of many workers at one (column group, round) --------------------------------------
// Philox4x32-10 at counter (q, worker, round, tag).  The parts of its first three rounds that do not depend
// on the worker are worked out once per (column group, round): of the twenty 32 x 32 -> 64 multiplies of a
// block sixteen remain per worker.  (A stream of such multiplies issues one per 5 cycles and
// scheduler; a block takes 65 of the 190 cycles of a row of a column group.  High halves by fp64 multiply-adds, whose
// pipe idles, took as long with 14 instructions more.)
struct NoiseBase {
  uint32_t a0, c3, c1, h0, l0;
};
__device__ __forceinline__ NoiseBase noise_base(uint32_t q, uint32_t round_lo, uint32_t ctr3, const PhiloxKeys& keys) {
  NoiseBase b;
  const uint64_t p0 = (uint64_t)kPhiloxMul0 * q, p1 = (uint64_t)kPhiloxMul1 * round_lo;
  b.a0 = (uint32_t)(p1 >> 32) ^ keys.k0[0];                       // with the worker word: word 0 after round 0
  const uint32_t c2 = (uint32_t)(p0 >> 32) ^ ctr3 ^ keys.k1[0];
  b.c3 = (uint32_t)p0 ^ keys.k1[1];
  const uint64_t q1 = (uint64_t)kPhiloxMul1 * c2;
  const uint32_t c0 = (uint32_t)(q1 >> 32) ^ (uint32_t)p1 ^ keys.k0[1];
  b.c1 = (uint32_t)q1 ^ keys.k0[2];
  const uint64_t p2 = (uint64_t)kPhiloxMul0 * c0;
  b.h0 = (uint32_t)(p2 >> 32) ^ keys.k1[2];
  b.l0 = (uint32_t)p2;
  return b;
}
// The same in two steps, for a thread that stays with a column group: what depends on neither worker nor round, and the rest.
struct NoiseColumn {
  uint32_t c3, h, c1;
};
__device__ __forceinline__ NoiseColumn noise_column(uint32_t q, uint32_t ctr3, const PhiloxKeys& keys) {
  const uint64_t p0 = (uint64_t)kPhiloxMul0 * q, q1 = (uint64_t)kPhiloxMul1 * ((uint32_t)(p0 >> 32) ^ ctr3 ^ keys.k1[0]);
  return NoiseColumn{(uint32_t)p0 ^ keys.k1[1], (uint32_t)(q1 >> 32) ^ keys.k0[1], (uint32_t)q1 ^ keys.k0[2]};
}
__device__ __forceinline__ NoiseBase noise_base(const NoiseColumn& c, uint32_t round_lo, const PhiloxKeys& keys) {
  NoiseBase b;
  const uint64_t p1 = (uint64_t)kPhiloxMul1 * round_lo, p2 = (uint64_t)kPhiloxMul0 * (c.h ^ (uint32_t)p1);
  b.a0 = (uint32_t)(p1 >> 32) ^ keys.k0[0];
  b.c3 = c.c3;
  b.c1 = c.c1;
  b.h0 = (uint32_t)(p2 >> 32) ^ keys.k1[2];
  b.l0 = (uint32_t)p2;
  return b;
}
// The one product that depends on worker and round alone.
__device__ __forceinline__ uint64_t noise_start(uint32_t worker, uint32_t round_lo, const PhiloxKeys& keys) {
  return (uint64_t)kPhiloxMul0 * (__umulhi(kPhiloxMul1, round_lo) ^ keys.k0[0] ^ worker);
}
// What noise_words takes when that product is given, from the low word of the round's product alone.
__device__ __forceinline__ NoiseBase noise_base_of_product(const NoiseColumn& c, uint32_t round_product, const PhiloxKeys& keys) {
  const uint64_t p2 = (uint64_t)kPhiloxMul0 * (c.h ^ round_product);
  return NoiseBase{0u, c.c3, c.c1, (uint32_t)(p2 >> 32) ^ keys.k1[2], (uint32_t)p2};
}
__device__ __forceinline__ uint4 noise_words(const NoiseBase& b, uint64_t e, const PhiloxKeys& keys) {
  const uint64_t p = (uint64_t)kPhiloxMul1 * ((uint32_t)(e >> 32) ^ b.c3);
  uint32_t c0 = (uint32_t)(p >> 32) ^ b.c1, c1 = (uint32_t)p, c2 = b.h0 ^ (uint32_t)e, c3 = b.l0;
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)kPhiloxMul0 * c0, p1 = (uint64_t)kPhiloxMul1 * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ keys.k0[r], n2 = (uint32_t)(p0 >> 32) ^ c3 ^ keys.k1[r];
    c0 = n0;
    c1 = (uint32_t)p1;
    c2 = n2;
    c3 = (uint32_t)p0;
  }
  return make_uint4(c0, c1, c2, c3);
}
__device__ __forceinline__ uint4 noise_words(const NoiseBase& b, uint32_t worker, const PhiloxKeys& keys) {
  return noise_words(b, (uint64_t)kPhiloxMul0 * (b.a0 ^ worker), keys);
}

}  // namespace netmax
