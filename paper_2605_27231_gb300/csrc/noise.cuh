// The N(0,1) draw of a lattice cell: Philox4x32-10 and a Box-Muller transform on two 53-bit uniforms.
//
// gauss_draw evaluates it in FP64 (the FP64 path).  gauss_draw_f32 gives the same number rounded to FP32 (the FP32
// path's noise) from pairs of FP32 values (an unevaluated sum hi + lo, about 48 bits): GB300 issues 64 FP32
// operations for one FP64 operation, and the FP64 logarithm, root and cosine of every cell were most of the synthesis
// (four USR realisations at 256^3: 9.5 -> 2.7 ms in all; one local one at 512^3: 20.6 -> 7.0 ms).  Both uniforms enter
// as the exact integers, and the argument reductions are exact, so the relative error of the pair before the final
// rounding is below 2^-30 everywhere, also where the logarithm or the cosine is near zero (2e7 draws against extended
// precision: RMS error 0.288546 ulp of FP32, 0.288545 for the rounded FP64 value).
#pragma once
#ifdef __CUDACC__
#include <cuda_runtime.h>
#endif
#include <math.h>
#include <stdint.h>

namespace sigw {

#ifdef __CUDA_ARCH__
#define SIGW_MULHI32(a, b) __umulhi(a, b)
#define SIGW_CLZ64(a) __clzll((long long)(a))
#define SIGW_FMUL(a, b) __fmul_rn(a, b)  // a product that is not contracted into a later sum
#else
#define SIGW_FMUL(a, b) ((a) * (b))
#define SIGW_MULHI32(a, b) ((uint32_t)(((uint64_t)(a) * (b)) >> 32))
#define SIGW_CLZ64(a) __builtin_clzll(a)
#endif

// Philox4x32-10 (SC'11): counter (c0, c1, c2, c3), key (k0, k1); 10 rounds, Weyl key schedule between rounds.
__host__ __device__ __forceinline__ void philox10(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3, uint32_t k0,
                                                  uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = SIGW_MULHI32(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = SIGW_MULHI32(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
}

// The two 53-bit uniforms of cell `cell` (row-major linear index) and key `seed`, as integers: u1 = (a + 1) 2^-53 in
// (0, 1], u2 = b 2^-53 in [0, 1).
__host__ __device__ __forceinline__ void noise_words(uint32_t cell, uint64_t seed, uint64_t& a, uint64_t& b) {
  uint32_t c0 = cell, c1 = 0u, c2 = 0u, c3 = 0u;
  philox10(c0, c1, c2, c3, (uint32_t)(seed & 0xffffffffull), (uint32_t)(seed >> 32));
  a = ((((uint64_t)c0) << 32) | c1) >> 11;
  b = ((((uint64_t)c2) << 32) | c3) >> 11;
}

#ifdef __CUDACC__
__device__ __forceinline__ double gauss_draw(uint32_t cell, uint64_t seed) {
  uint64_t a, b;
  noise_words(cell, seed, a, b);
  const double u1 = ((double)a + 1.0) * 1.1102230246251565404e-16;  // 2^-53
  const double u2 = (double)b * 1.1102230246251565404e-16;
  return sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
}
#endif

// ---- pairs of FP32 values (error-free sums and products after Dekker and Knuth)
struct ff {
  float h, l;
};
__host__ __device__ __forceinline__ ff ff_fast(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}
__host__ __device__ __forceinline__ ff ff_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
__host__ __device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = SIGW_FMUL(a.h, b.h);
  return ff_fast(p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h));
}
__host__ __device__ __forceinline__ ff ff_add(ff a, ff b) {
  const ff s = ff_sum(a.h, b.h);
  return ff_fast(s.h, s.l + (a.l + b.l));
}
// The integer m > 0 as m 2^-64 2^(clz m): the 48 leading bits, in [1/2, 1).
__host__ __device__ __forceinline__ ff ff_mantissa(uint64_t m, int* lz) {
  *lz = SIGW_CLZ64(m);
  m <<= *lz;
  return {(float)(uint32_t)(m >> 40) * 5.9604644775390625e-8f, (float)(uint32_t)((m >> 16) & 0xffffffu) * 3.5527136788005009e-15f};
}
__host__ __device__ __forceinline__ float pow2f(int e) {  // 2^e, -126 <= e <= 127
  union {
    uint32_t u;
    float f;
  } v;
  v.u = (uint32_t)(e + 127) << 23;
  return v.f;
}

// sqrt(-2 ln u1) for u1 = A 2^-53, 1 <= A <= 2^53.  u1 = m 2^e with m in [1/sqrt2, sqrt2), f = m - 1 exact as an
// integer, ln(1 + f) = 2 atanh(s), s = f / (2 + f), |s| <= 0.172, by its odd power series.
__host__ __device__ __forceinline__ ff ff_radius(uint64_t A) {
  const int z = SIGW_CLZ64(A);
  const uint64_t m = A << z;  // u1 = m 2^-64 2^(11 - z)
  const bool up = m >= 0xB504F333F9DE6484ull;  // m 2^-64 >= 1/sqrt2: use it, else its double
  const uint64_t d = up ? 0ull - m : m - 0x8000000000000000ull;  // |f| 2^64 or 2^63
  const int e = up ? 11 - z : 10 - z;
  ff f = {0.f, 0.f};
  if (d) {
    int lz;
    f = ff_mantissa(d, &lz);
    const float sc = pow2f(up ? -lz : 1 - lz);
    f.h *= up ? -sc : sc;
    f.l *= up ? -sc : sc;
  }
  // s = f / (2 + f): quotient, its residual, one correction
  const ff den = ff_fast(2.f, f.h);
  const float dl = den.l + f.l, inv = 1.f / den.h;
  const float q = f.h * inv;
  const float res = fmaf(-q, dl, fmaf(-q, den.h, f.h) + f.l);
  const ff s = ff_fast(q, res * inv);
  const ff s2 = ff_mul(s, s);
  const float x = s2.h;
  // sum_k s^(2k) / (2k + 3): the k = 0 term as a pair, the rest in FP32
  const float tail = fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.f / 17.f, 1.f / 15.f), 1.f / 13.f), 1.f / 11.f),
                                          1.f / 9.f), 1.f / 7.f), 0.2f);
  const ff third = {0.3333333433f, -9.934107759e-9f};
  const float xt = SIGW_FMUL(x, tail);
  const ff P = ff_fast(third.h, xt);
  const ff poly = {P.h, P.l + (third.l + fmaf(x, tail, -xt))};
  const ff t = ff_mul(s2, poly);
  ff y = ff_mul(s, t);
  y = ff_add(s, y);  // atanh(s)
  const float fe = (float)e;
  const ff ln2h = {0.3465735912f, -9.523271061e-10f};  // ln 2 / 2
  const float ph = SIGW_FMUL(fe, ln2h.h);
  const ff el = {ph, fmaf(fe, ln2h.h, -ph) + fe * ln2h.l};
  y = ff_add(el, y);                     // (ln u1) / 2 <= 0
  const float yh = -4.f * y.h, yl = -4.f * y.l;  // -2 ln u1
  const float r = sqrtf(yh);
  if (r == 0.f) return {0.f, 0.f};
  return ff_fast(r, (fmaf(-r, r, yh) + yl) * (0.5f / r));
}

// cos(2 pi b 2^-53), 0 <= b < 2^53: the nearest quarter turn is taken off exactly, Taylor series on |angle| <= pi/4.
__host__ __device__ __forceinline__ ff ff_cos_turn(uint64_t b) {
  const uint32_t quad = (uint32_t)((b + (1ull << 50)) >> 51);  // nearest quarter turn, 0..4
  const int64_t r = (int64_t)(b - ((uint64_t)quad << 51));     // |r| <= 2^50
  const uint64_t ar = (uint64_t)(r < 0 ? -r : r);
  int lz;
  ff w = ff_mantissa(ar ? ar : 1, &lz);
  const float sc = ar ? pow2f(11 - lz) : 0.f;
  w = {w.h * sc, w.l * sc};                            // r 2^-53, its 48 leading bits
  const ff c = {6.283185482e+00f, -1.748455531e-07f};  // 2 pi
  const ff a = ff_mul(w, c);
  const ff a2 = ff_mul(a, a);
  const float x = a2.h;
  ff v;
  if (quad & 1) {  // sine: a (1 + a2 (-1/6 + a2 (1/120 - ...)))
    const float tail = fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, -7.64716373e-13f, 1.60590438e-10f), -2.50521084e-8f),
                                            2.75573192e-6f), -1.98412698e-4f), 8.33333333e-3f);
    const ff k = {-0.1666666716f, 4.967053879e-9f};
    const float xt = SIGW_FMUL(x, tail);
    const ff P = ff_fast(k.h, xt);
    const ff t = ff_mul(a2, ff{P.h, P.l + (k.l + fmaf(x, tail, -xt))});
    v = ff_add(a, ff_mul(a, t));
    if (r < 0) v = {-v.h, -v.l};
    if (quad == 1) v = {-v.h, -v.l};  // cos(pi/2 + a) = -sin a, cos(3 pi/2 + a) = sin a
  } else {  // cosine: 1 + a2 (-1/2 + a2 (1/24 + a2 (-1/720 + ...)))
    const float tail = fmaf(x, fmaf(x, fmaf(x, fmaf(x, -1.14707456e-11f, 2.08767570e-9f), -2.75573192e-7f),
                                    2.48015873e-5f), -1.38888889e-3f);
    const ff k = {0.04166666791f, -1.241763470e-9f};
    const float xt = SIGW_FMUL(x, tail);
    const ff P = ff_fast(k.h, xt);
    ff t = ff_mul(a2, ff{P.h, P.l + (k.l + fmaf(x, tail, -xt))});
    t = ff_add(ff{-0.5f, 0.f}, t);
    t = ff_mul(a2, t);
    v = ff_add(ff{1.f, 0.f}, t);
    if (quad == 2) v = {-v.h, -v.l};
  }
  return v;
}

__host__ __device__ __forceinline__ float gauss_f32(uint64_t a, uint64_t b) {
  const ff r = ff_radius(a + 1), c = ff_cos_turn(b);
  const float p = SIGW_FMUL(r.h, c.h);
  return p + (fmaf(r.h, c.h, -p) + fmaf(r.h, c.l, r.l * c.h));
}
__host__ __device__ __forceinline__ float gauss_draw_f32(uint32_t cell, uint64_t seed) {
  uint64_t a, b;
  noise_words(cell, seed, a, b);
  return gauss_f32(a, b);
}

}  // namespace sigw
