// Device modular arithmetic for RNS limbs held in 64-bit words.
//
// Primes q satisfy 2^(k-1) < q < 2^k with k <= 62, so 4q fits a word and the
// transforms can keep lazy residues in [0, 4q) (Harvey's butterfly). The GPU
// has no 64x64 multiplier: every product below compiles to 32-bit
// IMAD.WIDE/IMAD.HI sequences, so the code keeps the number of wide products
// minimal:
//   * Shoup product with a precomputed companion w' = floor(w 2^64 / q):
//     one high product, two low products, one conditional subtract.
//   * Barrett reduction of a value x < 2^(63+k) (a product or a lazy sum of
//     products) with mu = floor(2^(63+k) / q):
//       qhat = hi64((x >> (k-1)) * mu),  r = x - qhat q in [0, 3q).
#pragma once
#include <cstdint>

typedef uint64_t u64;
typedef unsigned __int128 u128;

struct Modulus {
  u64 q;
  u64 mu;     // floor(2^(63+k) / q)
  int kbits;  // bit length of q
  int pad;
  u64 qinv;   // -q^-1 mod 2^64 (Montgomery reduction)
};

__device__ __forceinline__ u64 mulhi64(u64 a, u64 b) { return __umul64hi(a, b); }

// x = (hi, lo) < 2^(63+k)  ->  x mod q in [0, q)
__device__ __forceinline__ u64 barrett_reduce128(u64 hi, u64 lo, const Modulus& m) {
  int s = m.kbits - 1;
  u64 xs = (lo >> s) | (hi << (64 - s));  // s in [1, 61]
  u64 qh = mulhi64(xs, m.mu);
  u64 r = lo - qh * m.q;
  if (r >= m.q) r -= m.q;
  if (r >= m.q) r -= m.q;
  return r;
}

__device__ __forceinline__ u64 mul_mod(u64 a, u64 b, const Modulus& m) {
  return barrett_reduce128(mulhi64(a, b), a * b, m);
}

// Montgomery reduction: x = (hi, lo) < q 2^64 -> x 2^-64 mod q in [0, q).
// With m = lo * qinv mod 2^64, x + m q is divisible by 2^64; the low words
// cancel with a carry exactly when lo != 0, and (x + m q) / 2^64 < 2q.
__device__ __forceinline__ u64 redc128(u64 hi, u64 lo, u64 q, u64 qinv) {
  const u64 m = lo * qinv;
  const u64 t = hi + mulhi64(m, q) + (lo != 0 ? 1 : 0);
  return t >= q ? t - q : t;
}

// 128-bit accumulator of products; reduce once at the end.
struct Acc128 {
  u64 lo, hi;
  __device__ __forceinline__ void zero() { lo = 0; hi = 0; }
  __device__ __forceinline__ void mac(u64 a, u64 b) {
    u64 l = a * b, h = mulhi64(a, b);
    lo += l;
    hi += h + (lo < l ? 1 : 0);
  }
  // the same product-accumulate through the compiler's 128-bit arithmetic
  __device__ __forceinline__ void mac_wide(u64 a, u64 b) {
    const u128 s = (((u128)hi << 64) | lo) + (u128)a * b;
    lo = (u64)s;
    hi = (u64)(s >> 64);
  }
  __device__ __forceinline__ void add(u64 a) {
    lo += a;
    hi += (lo < a ? 1 : 0);
  }
};

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
  u64 s = a + b;
  return s >= q ? s - q : s;
}

__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// a * w mod q, result in [0, 2q); any a < 2^64, w < q.
__device__ __forceinline__ u64 shoup_lazy(u64 a, u64 w, u64 wp, u64 q) {
  u64 qh = mulhi64(a, wp);
  return a * w - qh * q;
}

__device__ __forceinline__ u64 shoup(u64 a, u64 w, u64 wp, u64 q) {
  u64 r = shoup_lazy(a, w, wp, q);
  return r >= q ? r - q : r;
}

// a * w mod q by halves, result in [0, 6q) for any a < 2^64 and q < 2^55:
// w0 = w, w1 = 2^32 w mod q, p0 and p1 = floor(w0 2^31 / q) and floor(w1 2^31 / q),
// nq2 = -2q mod 2^64. With a = h 2^32 + l, a w = l w0 + h w1 (mod q); Q = the
// high word of l p0 + h p1 (< 2^64) is less than 3 below (l w0 + h w1) / 2q and
// fits 32 bits; r = l w0 + h w1 - 2q Q, of which only the low 64 bits are formed.
// Written as multiply-add-with-carry pairs: ptxas turns each lo/hi pair into one
// 64-bit accumulating multiply, where the same sums of 64-bit C products become
// separate multiplies and adds (register-only forward butterflies on sm_103a:
// 13.1 instructions and 30.2 cycles a warp, against 15.9 and 33.5).
__device__ __forceinline__ u64 half_mul(u64 a, u64 w0, u64 w1, uint32_t p0, uint32_t p1, u64 nq2) {
  const uint32_t l = (uint32_t)a, h = (uint32_t)(a >> 32);
  uint32_t r0, r1;
  asm("{\n\t"
      ".reg .u32 t, k;\n\t"
      "mul.lo.u32 t, %2, %8;\n\t"
      "mul.hi.u32 k, %2, %8;\n\t"
      "mad.lo.cc.u32 t, %3, %9, t;\n\t"
      "madc.hi.u32 k, %3, %9, k;\n\t"
      "mul.lo.u32 %0, %2, %4;\n\t"
      "mul.hi.u32 %1, %2, %4;\n\t"
      "mad.lo.cc.u32 %0, %3, %6, %0;\n\t"
      "madc.hi.u32 %1, %3, %6, %1;\n\t"
      "mad.lo.cc.u32 %0, k, %10, %0;\n\t"
      "madc.hi.u32 %1, k, %10, %1;\n\t"
      "mad.lo.u32 %1, %2, %5, %1;\n\t"
      "mad.lo.u32 %1, %3, %7, %1;\n\t"
      "mad.lo.u32 %1, k, %11, %1;\n\t"
      "}"
      : "=&r"(r0), "=&r"(r1)
      : "r"(l), "r"(h), "r"((uint32_t)w0), "r"((uint32_t)(w0 >> 32)), "r"((uint32_t)w1), "r"((uint32_t)(w1 >> 32)),
        "r"(p0), "r"(p1), "r"((uint32_t)nq2), "r"((uint32_t)(nq2 >> 32)));
  return ((u64)r1 << 32) | r0;
}
