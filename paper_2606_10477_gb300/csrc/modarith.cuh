// Device modular arithmetic on 64-bit words, primes 1.5 2^32 <= q < 2^60.1 (33 to 60 bits, see h_prime_chain).
//
//  * Shoup multiplication by a fixed operand w with companion
//    w' = floor(w * 2^64 / q): result in [0, 2q) for any 64-bit input
//    (Shoup; bound as in Harvey, "Faster arithmetic for number-theoretic
//    transforms", 2014).
//  * Montgomery steps by 2^32 (Montgomery 1985) on 96-bit sums, see mont_mul_lazy and reduce128.
//  * Barrett reduction of a value x < q^2 with mu = floor(2^(2b) / q),
//    b = bit length of q (Barrett 1986): quotient estimate
//    floor(floor(x / 2^(b-1)) * mu / 2^(b+1)), remainder in [0, 3q).
#pragma once
#include <cstdint>

namespace hedap {

typedef uint64_t u64;
constexpr u64 kMinPrime = 3ull << 31;  // reduce_lazy's estimate; h_prime_dev refuses smaller ones

struct PrimeDev {  // per-prime constants used by the kernels
  u64 q;
  u64 mu;       // floor(2^(2b) / q)
  int b;        // bit length of q
  uint32_t nqi; // -q^-1 mod 2^32 (mont_mul_lazy)
  uint32_t rc;  // floor(2^64 / q) (reduce_lazy; q > 2^32)
  uint32_t pad;
  u64 r64, r96, r128;  // 2^64, 2^96, 2^128 mod q
};

// High 64 bits of x * y, exact, from 32-bit pieces: the middle column (hi(x0 y0) + lo(x0 y1) +
// lo(x1 y0)) is summed only for its carries, then the upper columns with carry chains.  Eight
// 32-bit multiply-adds; measured faster than four 32 x 32 -> 64 products with 64-bit partial sums.
__device__ __forceinline__ u64 mulhi64(u64 x, u64 y) {
  u64 h;
  asm("{\n\t"
      ".reg .u32 x0, x1, y0, y1, t0, t1, t2, h0, h1;\n\t"
      "mov.b64 {x0, x1}, %1;\n\t"
      "mov.b64 {y0, y1}, %2;\n\t"
      "mul.hi.u32 t0, x0, y0;\n\t"
      "mad.lo.cc.u32 t0, x0, y1, t0;\n\t"
      "madc.hi.u32 t1, x0, y1, 0;\n\t"
      "mad.lo.cc.u32 t0, x1, y0, t0;\n\t"
      "madc.hi.cc.u32 t1, x1, y0, t1;\n\t"
      "addc.u32 t2, 0, 0;\n\t"
      "mad.lo.cc.u32 h0, x1, y1, t1;\n\t"
      "madc.hi.u32 h1, x1, y1, t2;\n\t"
      "mov.b64 %0, {h0, h1};\n\t"
      "}"
      : "=l"(h)
      : "l"(x), "l"(y));
  return h;
}
// x * w - floor(x * wp / 2^64) * q  mod 2^64, in [0, 2q): the quotient qh = mulhi64(x, wp), then
// x * w + qh * (2^64 - q) mod 2^64 in two wide and four low multiply-adds.
__device__ __forceinline__ u64 shoup_mul_lazy(u64 x, u64 w, u64 wp, u64 q) {
  const u64 nq = 0 - q, qh = mulhi64(x, wp);
  u64 r;
  asm("{\n\t"
      ".reg .u32 x0, x1, a0, a1, n0, n1, h0, h1, r0, r1;\n\t"
      ".reg .u64 p;\n\t"
      "mov.b64 {x0, x1}, %1;\n\t"
      "mov.b64 {a0, a1}, %2;\n\t"
      "mov.b64 {n0, n1}, %4;\n\t"
      "mov.b64 {h0, h1}, %3;\n\t"
      "mul.wide.u32 p, a0, x0;\n\t"
      "mad.wide.u32 p, h0, n0, p;\n\t"
      "mov.b64 {r0, r1}, p;\n\t"
      "mad.lo.u32 r1, a0, x1, r1;\n\t"
      "mad.lo.u32 r1, a1, x0, r1;\n\t"
      "mad.lo.u32 r1, h0, n1, r1;\n\t"
      "mad.lo.u32 r1, h1, n0, r1;\n\t"
      "mov.b64 %0, {r0, r1};\n\t"
      "}"
      : "=l"(r)
      : "l"(x), "l"(w), "l"(qh), "l"(nq));
  return r;
}
// x * w mod q, lazily, for a fixed operand w held as the pair (a, b) = (w 2^32 mod q, w 2^64 mod q):
// with x = x1 2^32 + x0, x0 a + x1 b = x w 2^32 (mod q) is a 96-bit sum of four 32 x 32 -> 64 products,
// and one Montgomery step (Montgomery 1985: m = -r q^-1 mod 2^32, (r + m q) / 2^32) of two more brings it
// below (2 + x / 2^64) q: six wide products and one low one, against three wide, one high, two wide and
// four low ones of shoup_mul_lazy.  Any 64-bit x, odd q < 2^61.  The carries out of the low column are
// added into the high column, which stays below 2^64 (three products below 2^61.1, 2^61.1 and 2^61).
// The 64-bit sums around the carry chains are plain C so that the compiler may merge them with the caller's.
__device__ __forceinline__ u64 mont_mul_lazy(u64 x, u64 a, u64 b, u64 q, uint32_t nqi) {
  const uint32_t x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32), b0 = (uint32_t)b, q0 = (uint32_t)q;
  u64 p, c;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(x0), "r"((uint32_t)a));
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(c) : "r"(x0), "r"((uint32_t)(a >> 32)));
  asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c) : "r"(x1), "r"((uint32_t)(b >> 32)));
  uint32_t p0 = (uint32_t)p, p1 = (uint32_t)(p >> 32), c1 = (uint32_t)(c >> 32);
  asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\tmadc.hi.cc.u32 %1, %3, %4, %1;\n\taddc.u32 %2, %2, 0;"
      : "+r"(p0), "+r"(p1), "+r"(c1)
      : "r"(x1), "r"(b0));
  const uint32_t m = p0 * nqi;
  asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\tmadc.hi.cc.u32 %1, %3, %4, %1;\n\taddc.u32 %2, %2, 0;"
      : "+r"(p0), "+r"(p1), "+r"(c1)
      : "r"(m), "r"(q0));
  c = ((u64)c1 << 32) | (uint32_t)c;
  asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c) : "r"(m), "r"((uint32_t)(q >> 32)));
  return c + p1;
}
// x - k when the high word of x is above that of k: brings x below max(k + 2^32, x - k) with one comparison
// and two predicated subtractions (k a multiple of a modulus; the 2^32 are slack in the caller's bound)
__device__ __forceinline__ u64 sub_if_above(u64 x, u64 k) {
  asm("{\n\t"
      ".reg .pred p;\n\t"
      ".reg .u32 x0, x1, k0, k1;\n\t"
      "mov.b64 {x0, x1}, %0;\n\t"
      "mov.b64 {k0, k1}, %1;\n\t"
      "setp.gt.u32 p, x1, k1;\n\t"
      "@p sub.cc.u32 x0, x0, k0;\n\t"
      "@p subc.u32 x1, x1, k1;\n\t"
      "mov.b64 %0, {x0, x1};\n\t"
      "}"
      : "+l"(x)
      : "l"(k));
  return x;
}
// The same sum of four products kept open, so that several terms x_t w_t share one Montgomery step:
// columns p (weight 1) and c (weight 2^32, which takes p's carries); up to 6 terms for q < 2^60.1 (each adds at
// most 2^61 to c).  mont_finish returns less than (1 + sum over the terms of (1 + x_t / 2^64)) q.
struct MontAcc {
  u64 p, c;
};
__device__ __forceinline__ void mont_mac(MontAcc& s, u64 x, u64 a, u64 b) {
  asm("{\n\t"
      ".reg .u32 x0, x1, a0, a1, b0, b1, p0, p1, c0, c1;\n\t"
      ".reg .u64 c;\n\t"
      "mov.b64 {x0, x1}, %2;\n\t"
      "mov.b64 {a0, a1}, %3;\n\t"
      "mov.b64 {b0, b1}, %4;\n\t"
      "mov.b64 {p0, p1}, %0;\n\t"
      "mad.wide.u32 c, x0, a1, %1;\n\t"
      "mad.wide.u32 c, x1, b1, c;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "mad.lo.cc.u32 p0, x0, a0, p0;\n\t"
      "madc.hi.cc.u32 p1, x0, a0, p1;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mad.lo.cc.u32 p0, x1, b0, p0;\n\t"
      "madc.hi.cc.u32 p1, x1, b0, p1;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mov.b64 %0, {p0, p1};\n\t"
      "mov.b64 %1, {c0, c1};\n\t"
      "}"
      : "+l"(s.p), "+l"(s.c)
      : "l"(x), "l"(a), "l"(b));
}
// the open sum plus x itself (w = 1: a = 2^32, b = 2^64 mod q = r64): two products
__device__ __forceinline__ void mont_add(MontAcc& s, u64 x, u64 r64) {
  asm("{\n\t"
      ".reg .u32 x0, x1, b0, b1, p0, p1, c0, c1;\n\t"
      ".reg .u64 c;\n\t"
      "mov.b64 {x0, x1}, %2;\n\t"
      "mov.b64 {b0, b1}, %3;\n\t"
      "mov.b64 {p0, p1}, %0;\n\t"
      "mad.wide.u32 c, x1, b1, %1;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "add.cc.u32 c0, c0, x0;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mad.lo.cc.u32 p0, x1, b0, p0;\n\t"
      "madc.hi.cc.u32 p1, x1, b0, p1;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mov.b64 %0, {p0, p1};\n\t"
      "mov.b64 %1, {c0, c1};\n\t"
      "}"
      : "+l"(s.p), "+l"(s.c)
      : "l"(x), "l"(r64));
}
__device__ __forceinline__ u64 mont_finish(const MontAcc& s, u64 q, uint32_t nqi) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 q0, q1, p0, p1, c0, c1, m;\n\t"
      ".reg .u64 c;\n\t"
      "mov.b64 {p0, p1}, %1;\n\t"
      "mov.b64 {c0, c1}, %2;\n\t"
      "mov.b64 {q0, q1}, %3;\n\t"
      "mul.lo.u32 m, p0, %4;\n\t"
      "mad.lo.cc.u32 p0, m, q0, p0;\n\t"
      "madc.hi.cc.u32 p1, m, q0, p1;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mov.b64 c, {c0, c1};\n\t"
      "mad.wide.u32 c, m, q1, c;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "add.cc.u32 c0, c0, p1;\n\t"
      "addc.u32 c1, c1, 0;\n\t"
      "mov.b64 %0, {c0, c1};\n\t"
      "}"
      : "=l"(r)
      : "l"(s.p), "l"(s.c), "l"(q), "r"(nqi));
  return r;
}
// x - floor(estimate of x / q) q in [0, 2q) for q >= 1.5 2^32 with x / 2^64 + 2^32 / q < 1: the estimate
// floor(x1 rc / 2^32), x1 the high word and rc = floor(2^64 / q), is below x / q by less than
// 1 + 2^32 / q + x / 2^64 < 2
__device__ __forceinline__ u64 reduce_lazy(u64 x, u64 q, uint32_t rc) {
  const uint32_t h = __umulhi((uint32_t)(x >> 32), rc);
  return x - h * q;
}
__device__ __forceinline__ u64 shoup_mul(u64 x, u64 w, u64 wp, u64 q) {
  u64 r = shoup_mul_lazy(x, w, wp, q);
  return r >= q ? r - q : r;
}
__device__ __forceinline__ u64 barrett_reduce(u64 lo, u64 hi, const PrimeDev& p) {
  // t = floor(x / 2^(b-1)) (< 2^(b+1)), qhat = floor(t * mu / 2^(b+1))
  int s = p.b - 1;
  u64 t = (lo >> s) | (hi << (64 - s));
  u64 plo = t * p.mu, phi = mulhi64(t, p.mu);
  int s2 = p.b + 1;
  u64 qhat = (plo >> s2) | (phi << (64 - s2));
  u64 r = lo - qhat * p.q;
  if (r >= p.q) r -= p.q;
  if (r >= p.q) r -= p.q;
  return r;
}
__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
  u64 s = a + b;
  return s >= q ? s - q : s;
}
__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) {
  return a >= b ? a - b : a + q - b;
}
// 128-bit accumulator helpers for lazy sums of products
struct Acc128 {
  u64 lo, hi;
};
// acc += a * b (the caller keeps the sum below 2^128): the products of equal halves go to the accumulator's two
// aligned register pairs, the cross products are summed apart (a, b with a1 b0 + a0 b1 < 2^64, i.e. a < 2^63.8 with
// b < 2^57, or both below 2^61.9) and added across the pairs.  Four wide products and three additions; as four 32-bit
// columns in one carry chain the cross products straddled the pairs and cost a low and a high product each.
__device__ __forceinline__ void mac128(Acc128& acc, u64 a, u64 b) {
  asm("{\n\t"
      ".reg .u32 a0, a1, b0, b1, c0, c1, c2, c3, m0, m1;\n\t"
      ".reg .u64 m;\n\t"
      "mov.b64 {a0, a1}, %2;\n\t"
      "mov.b64 {b0, b1}, %3;\n\t"
      "mov.b64 {c0, c1}, %0;\n\t"
      "mov.b64 {c2, c3}, %1;\n\t"
      "mul.wide.u32 m, a0, b1;\n\t"
      "mad.wide.u32 m, a1, b0, m;\n\t"
      "mov.b64 {m0, m1}, m;\n\t"
      "mad.lo.cc.u32 c0, a0, b0, c0;\n\t"
      "madc.hi.cc.u32 c1, a0, b0, c1;\n\t"
      "madc.lo.cc.u32 c2, a1, b1, c2;\n\t"
      "madc.hi.u32 c3, a1, b1, c3;\n\t"
      "add.cc.u32 c1, c1, m0;\n\t"
      "addc.cc.u32 c2, c2, m1;\n\t"
      "addc.u32 c3, c3, 0;\n\t"
      "mov.b64 %0, {c0, c1};\n\t"
      "mov.b64 %1, {c2, c3};\n\t"
      "}"
      : "+l"(acc.lo), "+l"(acc.hi)
      : "l"(a), "l"(b));
}
__device__ __forceinline__ Acc128 mul128(u64 a, u64 b) {  // a, b < 2^61
  Acc128 r;
  asm("{\n\t"
      ".reg .u32 a0, a1, b0, b1, c0, c1, c2, c3, m0, m1;\n\t"
      ".reg .u64 m, p;\n\t"
      "mov.b64 {a0, a1}, %2;\n\t"
      "mov.b64 {b0, b1}, %3;\n\t"
      "mul.wide.u32 m, a0, b1;\n\t"
      "mad.wide.u32 m, a1, b0, m;\n\t"
      "mov.b64 {m0, m1}, m;\n\t"
      "mul.wide.u32 p, a0, b0;\n\t"
      "mov.b64 {c0, c1}, p;\n\t"
      "mul.wide.u32 p, a1, b1;\n\t"
      "mov.b64 {c2, c3}, p;\n\t"
      "add.cc.u32 c1, c1, m0;\n\t"
      "addc.cc.u32 c2, c2, m1;\n\t"
      "addc.u32 c3, c3, 0;\n\t"
      "mov.b64 %0, {c0, c1};\n\t"
      "mov.b64 %1, {c2, c3};\n\t"
      "}"
      : "=l"(r.lo), "=l"(r.hi)
      : "l"(a), "l"(b));
  return r;
}
// canonical residue of any 128-bit value x = hi 2^64 + lo: hi by mont_mac's pair (2^96, 2^128) of 2^64, plus lo, in
// one Montgomery step (below 5q), then three conditional subtractions.  Nine wide products, against about
// twenty-five of two Barrett reductions and a Shoup product.
__device__ __forceinline__ u64 reduce128(Acc128 x, const PrimeDev& p) {
  MontAcc s{0, 0};
  mont_mac(s, x.hi, p.r96, p.r128);
  mont_add(s, x.lo, p.r64);
  u64 r = mont_finish(s, p.q, p.nqi);
  if (r >= p.q * 4) r -= p.q * 4;
  if (r >= p.q * 2) r -= p.q * 2;
  return r >= p.q ? r - p.q : r;
}
__device__ __forceinline__ u64 mul_mod(u64 a, u64 b, const PrimeDev& p) { return reduce128(mul128(a, b), p); }

}  // namespace hedap
