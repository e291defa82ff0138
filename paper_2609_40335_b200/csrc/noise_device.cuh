// Device-side Gaussian stream shared by the stand-alone noise kernel and the GEMM epilogue.
//
// z_j is a pure function of (seed, tensor_id, step, j): Philox4x32 with 10 rounds, key =
// (seed low, seed high), counter = (j/4 low, j/4 high, tensor_id, step); the four output
// words give four normals by Box-Muller on the word pairs (x0,x1) and (x2,x3):
//   u1 = ((xa >> 8) + 1) * 2^-24 in (0,1],  u2 = (xb >> 8) * 2^-24 in [0,1)   (exact in fp32)
//   r = sqrt(-2 ln u1),  z = r cos(2 pi u2),  r sin(2 pi u2).
//
// The generator is bound by the ALU and FMA pipes wherever it runs, so it is written for the 24-bit
// integers it gets: no special cases, no branch on the common path, both pairs of a counter side by
// side in packed fp32x2 operations, the Philox round keys expanded on the host (constant operands).
//   radius     256 k = 2^e m with m in [11/16, 11/8), k = 2^24 u1, g = 2 - 2m (exact):
//              t = -2 ln u1 = -2 ln 2 * (e - 32) + g + g^2 R(g), R a degree-7 minimax polynomial
//              (weighted least squares with Lawson's reweighting); sqrt(t) as rh + rl: reciprocal
//              square root and one Newton step whose correction rl is never rounded into rh.
//   direction  2 pi u2 = pi/2 * (quadrant + y), |y| <= 1/2: the top two bits of xb + 2^29 are the
//              quadrant, the next 22 go straight into a float's mantissa; minimax polynomials for
//              sin and cos of pi/2 * y, swapped by the quadrant, its sign carried by the radius.
// Measured (38.6 M elements, idle boost clock): add 413 -> 536, fill 428 -> 595 G elements/s against
// logf / sqrt / sincospif one pair at a time; 61 -> 39 instructions per element, the heavy half of the
// FMA pipe (20 wide multiplies of Philox, the packed FMAs) 71 % busy.
//
// Accuracy: an exhaustive scan over all 2^24 inputs of each factor (dp_debug_noise_error_scan,
// checked by a GPU test) gives max relative error 4.7e-8 for the radius and max absolute error
// 5.9e-8 for the cosine / sine (9.6e-8 and 5.3e-8 before); with the 2^-24 rounding of the product
// the error of z is at most r * 1.7e-7, 7.5e-7 at r = 4.5.  Pairs with a larger radius (4e-5 of
// them) take a float64 path, whose only error is the final rounding to fp32.
#pragma once

#include <stdint.h>

namespace dpg {

// Philox round keys of one seed, expanded on the host.  Kept in kernel parameters: the unrolled
// rounds then read them as constant operands (no adds, no registers).
struct NoiseKeys {
  uint32_t k0[10], k1[10];
};
inline NoiseKeys expand_noise_keys(uint64_t seed) {
  NoiseKeys K;
  uint32_t a = uint32_t(seed), b = uint32_t(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    K.k0[r] = a; K.k1[r] = b;
    a += 0x9E3779B9u; b += 0xBB67AE85u;
  }
  return K;
}

// The step word of a launch: the host's value plus, when a device counter is registered
// (dp_noise_step_device), the counter's current value -- so that a captured CUDA graph draws
// fresh noise at every replay.
__device__ __forceinline__ uint32_t effective_step(uint32_t step, const uint32_t* step_dev) {
  return step_dev ? step + __ldg(step_dev) : step;
}

struct U4 { uint32_t x, y, z, w; };

__device__ __forceinline__ U4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                            const NoiseKeys& K) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // one 32x32->64 multiply per half round gives both product words
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
    const uint32_t hi0 = uint32_t(p0 >> 32), lo0 = uint32_t(p0);
    const uint32_t hi1 = uint32_t(p1 >> 32), lo1 = uint32_t(p1);
    c0 = hi1 ^ c1 ^ K.k0[r]; c1 = lo1; c2 = hi0 ^ c3 ^ K.k1[r]; c3 = lo0;
  }
  return U4{c0, c1, c2, c3};
}

// ---- packed fp32 pairs ------------------------------------------------------------------
struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ void unpack(F2 p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

// ---- Box-Muller factors -----------------------------------------------------------------
// t = -2 ln u1 of two words and its square root rh + rl, negated where the top bit of the matching
// v is set
__device__ __forceinline__ void bm_radius(uint32_t xa, uint32_t xc, uint32_t va, uint32_t vc,
                                          float& ta, float& tc, F2& rh, F2& rl) {
  constexpr int kLow = 0x3f300000 + (32 << 23);                // bits of 2^32 * 11/16
  float ka, kc;                                                // 256 ((x >> 8) + 1), exact
  unpack(add2(f2(float(xa & 0xffffff00u), float(xc & 0xffffff00u)), f2(256.f)), ka, kc);
  const int ba = __float_as_int(ka), bc = __float_as_int(kc);
  const int ea = (ba - kLow) & int(0xff800000), ec = (bc - kLow) & int(0xff800000);   // (e - 32) << 23
  const F2 g = fma2(f2(__int_as_float(ba - ea), __int_as_float(bc - ec)), f2(-0x1p-31f), f2(2.f));
  F2 p = f2(4.283334966e-04f);
  p = fma2(p, g, f2(1.176905195e-03f));
  p = fma2(p, g, f2(2.277112492e-03f));
  p = fma2(p, g, f2(5.145088168e-03f));
  p = fma2(p, g, f2(1.248652348e-02f));
  p = fma2(p, g, f2(3.125725262e-02f));
  p = fma2(p, g, f2(8.333430510e-02f));
  p = fma2(p, g, f2(2.499997878e-01f));
  const F2 t = fma2(f2(float(ea), float(ec)), f2(-1.652591664e-07f),      // -2 ln 2 / 2^23
                    fma2(mul2(g, g), p, g));
  unpack(t, ta, tc);
  ta = fmaxf(ta, 1e-30f);                                      // u1 = 1: r = 1e-15 stands for 0
  tc = fmaxf(tc, 1e-30f);
  float ya, yc;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ya) : "f"(ta));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yc) : "f"(tc));
  const F2 y = f2(__uint_as_float(__float_as_uint(ya) ^ (va & 0x80000000u)),
                  __uint_as_float(__float_as_uint(yc) ^ (vc & 0x80000000u)));
  const F2 tt = f2(ta, tc);
  rh = mul2(tt, y);
  rl = mul2(fma2(mul2(rh, f2(-0.5f)), rh, mul2(tt, f2(0.5f))), y);        // (t - rh^2) / (2 rh)
}

// cos and sin of 2 pi u2 for two words, given v = xb + 2^29, up to the sign in the top bit of v
__device__ __forceinline__ void bm_direction(uint32_t vb, uint32_t vd, F2& c, F2& s) {
  const F2 y = add2(f2(__uint_as_float(((vb >> 7) & 0x007ffffeu) | 0x3f800000u),
                       __uint_as_float(((vd >> 7) & 0x007ffffeu) | 0x3f800000u)), f2(-1.5f));
  const F2 y2 = mul2(y, y);
  F2 p = fma2(y2, f2(-4.600182095e-03f), f2(7.967966622e-02f));
  p = fma2(p, y2, f2(-6.459634771e-01f));
  p = fma2(p, y2, f2(-4.371138829e-08f));                      // low word of pi/2
  const F2 sn = fma2(y, f2(1.570796371f), mul2(y, p));
  F2 q = fma2(y2, f2(9.040186462e-04f), f2(-2.086028724e-02f));
  q = fma2(q, y2, f2(2.536692439e-01f));
  q = fma2(q, y2, f2(-1.233700543f));
  const F2 cs = fma2(q, y2, f2(1.f));
  float s0, s1, c0, c1;
  unpack(sn, s0, s1);
  unpack(cs, c0, c1);
  const bool swb = (vb & 0x40000000u) != 0, swd = (vd & 0x40000000u) != 0;      // odd quadrants
  c = f2(swb ? -s0 : c0, swd ? -s1 : c1);
  s = f2(swb ? c0 : s0, swd ? c1 : s1);
}

// the four normals of one counter's words, fp32 path; ta, tc: the squared radii
__device__ __forceinline__ void box_muller(const U4& x, float& z0, float& z1, float& z2, float& z3,
                                           float& ta, float& tc) {
  const uint32_t vb = x.y + 0x20000000u, vd = x.w + 0x20000000u;
  F2 rh, rl, c, s;
  bm_radius(x.x, x.z, vb, vd, ta, tc, rh, rl);
  bm_direction(vb, vd, c, s);
  unpack(fma2(rl, c, mul2(rh, c)), z0, z2);
  unpack(fma2(rl, s, mul2(rh, s)), z1, z3);
}

// fp32 path while r^2 stays below this; see above for how it follows from the measured error of the
// two factors
#ifndef DPG_NOISE_TAIL_T
#define DPG_NOISE_TAIL_T 20.25f
#endif

// the same whatever the radius: pairs beyond the threshold in float64.  Out of line: one warp in
// four hundred comes here.
static __device__ __noinline__ float4 box_muller_tail(U4 x) {
  const uint32_t a[2] = {x.x, x.z}, b[2] = {x.y, x.w};
  float o[4], t[2];
  box_muller(x, o[0], o[1], o[2], o[3], t[0], t[1]);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (t[h] > DPG_NOISE_TAIL_T) {
      const double r = sqrt(-2.0 * log(double((a[h] >> 8) + 1u) * 5.9604644775390625e-08));
      double sd, cd;
      sincospi(double(b[h] >> 8) * 1.1920928955078125e-07, &sd, &cd);
      o[2 * h] = float(r * cd);
      o[2 * h + 1] = float(r * sd);
    }
  }
  return make_float4(o[0], o[1], o[2], o[3]);
}

// the four normals of counter q (elements 4q .. 4q+3 of the tensor)
__device__ __forceinline__ void normals4(unsigned long long q, const NoiseKeys& K, uint32_t tensor_id,
                                         uint32_t step, float (&z)[4]) {
  const U4 x = philox4x32_10(uint32_t(q), uint32_t(q >> 32), tensor_id, step, K);
  float ta, tc;
  box_muller(x, z[0], z[1], z[2], z[3], ta, tc);
  if (fmaxf(ta, tc) > DPG_NOISE_TAIL_T) {
    const float4 f = box_muller_tail(x);
    z[0] = f.x; z[1] = f.y; z[2] = f.z; z[3] = f.w;
  }
}

// Eq. 3 on one element: scale * (v + amp * z)
__device__ __forceinline__ float noised(float v, float z, float amp, float scale) {
  return scale * fmaf(amp, z, v);
}

}  // namespace dpg
