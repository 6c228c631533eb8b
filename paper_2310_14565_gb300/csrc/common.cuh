// Shared device types and modular arithmetic for the PEPSI GB300 library.
//
// Modular reduction follows published methods, written from their
// definitions:
//  - Shoup's precomputed-quotient multiplication (NTL) for a fixed operand w:
//    w' = floor(w 2^64 / q); r = w x - umulhi(w', x) q lies in [0, 2q).
//  - Barrett reduction (Barrett 1986): of a product of two values below
//    2^bits(q) with the one-word constant floor(2^(bits+63) / q), and of a
//    64-bit value with floor(2^64 / q); a 128-bit value as hi (2^64 mod q)
//    (Shoup) plus lo (Barrett).
//  - Harvey's lazy butterflies (Harvey 2014) keep NTT values in [0, 4q).
// All primes are below 2^61, so 4q < 2^63 and every lazy sum fits in 64 bits.
#pragma once
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

typedef uint64_t u64;
typedef uint32_t u32;
typedef int64_t i64;

#define PEPSI_MAXQ 8   // ciphertext primes q_i
#define PEPSI_MAXB 12  // auxiliary primes p_j of the exact multiplication base
#define PEPSI_MAXP (PEPSI_MAXQ + PEPSI_MAXB + 1)  // + the plaintext modulus t
#define PEPSI_DUMMY 0xFFFFFFFFFFFFFFFFull
#define PEPSI_CW_NONE 0xFFFFu

// One modulus q of n = bits(q) bits (n <= 61): N^-1 (Shoup); the split point
// s = ceil(n/2) of the split operand format (hi << 32 | lo with x = hi 2^s +
// lo) used by the multiply-accumulate; and the reduction constants
// mu = floor(2^(n+63)/q), m64 = floor(2^64/q), c64 = 2^64 mod q (Shoup).
// pm: q = 2^n - d with d small enough for the folding products below (PmMul);
// the companion of a fixed operand w in the transform tables (and ninvs) is
// then w 2^s mod q instead of Shoup's quotient.
struct DevPrime {
  u64 q, ninv, ninvs, split, nbits, mu, m64, c64, c64s;
  u32 pm, d, s, pad;
};
__host__ __device__ __forceinline__ u64 to_split(u64 x, u64 s) { return ((x >> s) << 32) | (x & ((1ull << s) - 1)); }
__host__ __device__ __forceinline__ u64 from_split(u64 w, u64 s) { return ((w >> 32) << s) | (w & 0xFFFFFFFFull); }

// Constants of the exact RNS conversions (all residues reduced, companions
// where the value multiplies a varying operand: Shoup's, or with pm the folding
// products' for cq, qb, qinv_b, cb and bq).
struct RnsConst {
  u64 pm;  // every prime has folding products and their inputs fit (host.cpp)
  // Garner over Q: cq[i][j] = q_j^-1 mod q_i (j < i)
  u64 cq[PEPSI_MAXQ][PEPSI_MAXQ], cqs[PEPSI_MAXQ][PEPSI_MAXQ];
  // radices of Q in B for Horner's rule: qb[j][l] = q_l mod p_j (Shoup)
  u64 qb[PEPSI_MAXB][PEPSI_MAXQ], qbs[PEPSI_MAXB][PEPSI_MAXQ];
  u64 qhalf_dig[PEPSI_MAXQ];  // mixed-radix digits of (Q-1)/2 over Q
  u64 qmodb[PEPSI_MAXB];      // Q mod p_j
  u64 qhalf_b[PEPSI_MAXB];    // (Q-1)/2 mod p_j
  u64 qinv_b[PEPSI_MAXB], qinv_bs[PEPSI_MAXB];  // Q^-1 mod p_j
  u64 qhalf_q[PEPSI_MAXQ];    // (Q-1)/2 mod q_i
  u64 t_q[PEPSI_MAXQ], t_qs[PEPSI_MAXQ];        // t mod q_i
  u64 t_b[PEPSI_MAXB], t_bs[PEPSI_MAXB];        // t mod p_j
  // Garner over B
  u64 cb[PEPSI_MAXB][PEPSI_MAXB], cbs[PEPSI_MAXB][PEPSI_MAXB];
  u64 bq[PEPSI_MAXQ][PEPSI_MAXB], bqs[PEPSI_MAXQ][PEPSI_MAXB];  // p_l mod q_i (Shoup)
  u64 bhalf_dig[PEPSI_MAXB];        // mixed-radix digits of (B-1)/2 over B
  u64 bmodq[PEPSI_MAXQ];            // B mod q_i
  // decryption and encoding
  u64 pq_t[PEPSI_MAXQ];     // prod_{m<l} q_m mod t
  double pq_d[PEPSI_MAXQ];  // prod_{m<l} q_m as a double
  u64 qinv_t;               // Q^-1 mod t
  u64 qhalf_t;              // (Q-1)/2 mod t
  u64 qdt_q[PEPSI_MAXQ], qdt_qs[PEPSI_MAXQ];  // floor(Q/t) mod q_i
  u64 qmt;                  // Q mod t
};

// Primes (Q then B) and conversion constants passed by value to the exact
// RNS kernels, so that they are read from the kernel parameter space.
struct RnsArgs {
  DevPrime pr[PEPSI_MAXQ + PEPSI_MAXB];
  RnsConst rc;
  int N, k, kb;
};

// Everything a kernel needs to know about one parameter set.
struct DevView {
  int N, logN, k, kb, tidx;  // tidx: index of t among the moduli (= k + kb)
  const DevPrime* pr;        // [k + kb + 1]
  const ulonglong2* twp;     // [np][N] (psi^brev(i), its Shoup companion)
  const ulonglong2* itwp;    // [np][N] (psi^-brev(i), its Shoup companion); entry 0: psi^-brev(1) N^-1
  const RnsConst* rc;
  const RnsArgs* host_args;  // host copy for by-value launches (not dereferenced on the device)
  int allpm;                 // every ciphertext and auxiliary prime has folding products (kernels' PM forms)
  int nt;                    // threads per block of the ciphertext transforms (0: the default for N)
};
// The rings a transform kernel is compiled for: all, or those below N = 4096 alone.
// The named barriers of the fused forms (N = 4096, 8192, 16384) reserve all sixteen of
// a block's barriers, which limits the small blocks of small rings: 1500 x 4 rows of N
// = 256 took 34 us in the kernels with the fused forms and 16 us without, N = 1024 66
// and 51 us.  Kernels for 4096 and up alone, without the generic form, were slower by
// up to 1 % (they spilled more).
enum Ring { RING_ANY, RING_SMALL };
constexpr int FUSED_LOGN = 12;


// ---------------------------------------------------------------- arithmetic
__device__ __forceinline__ u64 shoup_lazy(u64 x, u64 w, u64 ws, u64 q) {
  u64 qh = __umul64hi(x, ws);
  return x * w - qh * q;  // in [0, 2q)
}
__device__ __forceinline__ u64 shoup(u64 x, u64 w, u64 ws, u64 q) {
  u64 r = shoup_lazy(x, w, ws, q);
  return r >= q ? r - q : r;
}
// Products by a fixed w modulo q = 2^n - d (the primes are the largest below a
// power of two, so d is small).  With v = w 2^s mod q, s = ceil((n + 5) / 2), and
// x = x1 2^s + x0 < 2^(n+5): x w = x0 w + x1 v (mod q), a sum S below 2^(n+s+1)
// of four 32-bit wide products, and 2^n = d folds its top: S mod 2^n + floor(S /
// 2^n) d < 2 q, one more product.  Five wide products (the quarter-rate
// operation that bounds the transforms) against the eight or so of Shoup's method
// (a 64-bit high product and two low ones): 32 against 41 cycles a warp for a
// butterfly in registers.
struct PmMul {
  u64 q;
  u32 d, s, n32, smask, nmask;
  __device__ __forceinline__ explicit PmMul(const DevPrime& p)
      : q(p.q), d(p.d), s(p.s), n32((u32)p.nbits - 32), smask((1u << p.s) - 1), nmask((1u << (p.nbits - 32)) - 1) {}
  // x < 2^(n+5) -> [0, 2q)
  __device__ __forceinline__ u64 mul(u64 x, u64 w, u64 v) const {
    const u32 x0 = (u32)x & smask, x1 = __funnelshift_r((u32)x, (u32)(x >> 32), s);
    u64 r;  // L = x0 wl + x1 vl < 2^(s+33) <= 2^64, M = x0 wh + x1 vh + (L >> 32)
    asm("{\n\t"
        ".reg .u64 L, M;\n\t.reg .u32 l, h, m, k, t;\n\t"
        "mul.wide.u32 L, %1, %3;\n\tmul.wide.u32 M, %1, %4;\n\t"
        "mad.wide.u32 L, %2, %5, L;\n\tmad.wide.u32 M, %2, %6, M;\n\t"
        "mov.b64 {l, h}, L;\n\tmov.b64 {m, k}, M;\n\t"
        "add.cc.u32 m, m, h;\n\taddc.u32 k, k, 0;\n\t"
        "shf.r.wrap.b32 t, m, k, %7;\n\tand.b32 m, m, %8;\n\t"
        "mov.b64 L, {l, m};\n\tmad.wide.u32 %0, t, %9, L;\n\t}"
        : "=l"(r)
        : "r"(x0), "r"(x1), "r"((u32)w), "r"((u32)(w >> 32)), "r"((u32)v), "r"((u32)(v >> 32)), "r"(n32), "r"(nmask),
          "r"(d));
    return r;
  }
  // x c for c < 2^32 and x c < 2^(n+32) -> below 2^n + 2^32 d
  __device__ __forceinline__ u64 mul_small(u64 x, u32 c) const {
    const u64 L = (u64)(u32)x * c, M = (u64)(u32)(x >> 32) * c + (L >> 32);
    return (u64)(u32)(M >> n32) * d + ((u64)((u32)M & nmask) << 32 | (u32)L);
  }
  // x < 2^(n+5) -> [0, 2^n + 2^32) with x = x1 2^n + x0: x0 + x1 d, x1 < 32, d < 2^27
  // (and x1 d < q, so one subtraction reduces it)
  __device__ __forceinline__ u64 fold(u64 x) const {
    const u32 h = (u32)(x >> 32);
    return ((u64)(h & nmask) << 32 | (u32)x) + (h >> n32) * d;
  }
};
// x mod q for any 64-bit x: one-word Barrett, floor(x m64 / 2^64) is short
// of floor(x/q) by at most 1.
__device__ __forceinline__ u64 barrett64(u64 x, const DevPrime& p) {
  const u64 r = x - __umul64hi(x, p.m64) * p.q;  // [0, 2q)
  return r >= p.q ? r - p.q : r;
}
// (hi:lo) mod q for any 128-bit value: hi 2^64 = hi c64 (mod q) by Shoup
// and lo by one-word Barrett, each in [0, 2q), then their sum reduced.
__device__ __forceinline__ u64 reduce128(u64 hi, u64 lo, const DevPrime& p) {
  const u64 a = shoup_lazy(hi, p.c64, p.c64s, p.q);
  const u64 b = lo - __umul64hi(lo, p.m64) * p.q;
  const u64 q2 = 2 * p.q;
  u64 r = a + b;  // [0, 4q)
  r = r >= q2 ? r - q2 : r;
  return r >= p.q ? r - p.q : r;
}
// a b mod q for a, b < 2^n (Barrett 1973, one constant): x = a b < 2^2n,
// x1 = floor(x / 2^(n-1)) < 2^(n+1), and floor(x1 mu / 2^64) is short of
// floor(x/q) by at most 2 (the dropped fractions are below 1/4 and 1).
__device__ __forceinline__ u64 mulmod(u64 a, u64 b, const DevPrime& p) {
  const u64 lo = a * b, hi = __umul64hi(a, b);
  const int n = (int)p.nbits;
  const u64 x1 = (hi << (65 - n)) | (lo >> (n - 1));
  u64 r = lo - __umul64hi(x1, p.mu) * p.q;  // [0, 3q)
  const u64 q2 = 2 * p.q;
  r = r >= q2 ? r - q2 : r;
  return r >= p.q ? r - p.q : r;
}
__device__ __forceinline__ u64 addmod(u64 a, u64 b, u64 q) {
  u64 s = a + b;
  return s >= q ? s - q : s;
}
__device__ __forceinline__ u64 submod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }
// (hi:lo) < 2^(2n+5) mod q = 2^n - d (a sum of up to 32 products of residues): two
// folds, three wide products against the six or so of Barrett's.  The condition of
// pm, 2^(s+1) d < 2^n with s >= (n + 5) / 2, gives d < 2^((n-7)/2), so the second fold's
// product, below 2^5 d^2, stays below 2^(n-2).
__device__ __forceinline__ u64 pm_reduce(u64 hi, u64 lo, const PmMul& m, int n) {
  const u64 h = hi << (64 - n) | lo >> n;
  const u64 low = (u64)((u32)(lo >> 32) & m.nmask) << 32 | (u32)lo;
  const u64 L = (u64)(u32)h * m.d, M = (u64)(u32)(h >> 32) * m.d + (L >> 32);  // h d = M 2^32 + L mod 2^32
  const u64 f = (u64)((u32)M & m.nmask) << 32 | (u32)L;
  u64 r = low + f + (u64)(u32)(M >> m.n32) * m.d;  // M / 2^(n-32) = h d / 2^n < 32 d < 2^32
  r = m.fold(r);
  return r >= m.q ? r - m.q : r;
}
// 128-bit accumulate acc += a*b
__device__ __forceinline__ void mac128(u64& lo, u64& hi, u64 a, u64 b) {
  asm("mad.lo.cc.u64 %0, %2, %3, %0;\n\tmadc.hi.u64 %1, %2, %3, %1;" : "+l"(lo), "+l"(hi) : "l"(a), "l"(b));
}
__device__ __forceinline__ u32 brev_bits(u32 x, int bits) { return bits ? (__brev(x) >> (32 - bits)) : 0; }

// ------------------------------------------------------------- SplitMix64
// Counter-based use of SplitMix64 (Steele, Lea, Flood 2014): the idx-th
// output of a generator whose state starts at mix64(seed ^ mix64(stream)).
#define PEPSI_GOLDEN 0x9E3779B97F4A7C15ull
__host__ __device__ __forceinline__ u64 mix64(u64 z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ u64 stream_key(u64 seed, u64 stream) { return mix64(seed ^ mix64(stream)); }
__host__ __device__ __forceinline__ u64 draw_keyed(u64 key, u64 idx) { return mix64(key + (idx + 1) * PEPSI_GOLDEN); }
// uniform in [0, bound) by rejection, attempt a at index pos*256 + a
__host__ __device__ __forceinline__ u64 sample_uniform(u64 key, u64 pos, u64 bound) {
  u64 rem = (0 - bound) % bound;
  u64 r = 0;
  for (u64 a = 0; a < 256; a++) {
    r = draw_keyed(key, (pos << 8) | a);
    if (rem == 0 || r < (u64)(0 - rem)) return r % bound;
  }
  return r % bound;
}
// centred binomial, eta = 21
__host__ __device__ __forceinline__ int sample_cbd21(u64 key, u64 pos) {
  u64 r = draw_keyed(key, pos);
#ifdef __CUDA_ARCH__
  return __popcll(r & 0x1FFFFFull) - __popcll((r >> 21) & 0x1FFFFFull);
#else
  return __builtin_popcountll(r & 0x1FFFFFull) - __builtin_popcountll((r >> 21) & 0x1FFFFFull);
#endif
}
__host__ __device__ __forceinline__ u64 make_stream(u64 purpose, u64 index, u64 prime) {
  return (purpose << 56) | (index << 8) | prime;
}
enum { STREAM_SK = 1, STREAM_RLK_A = 2, STREAM_RLK_E = 3, STREAM_ENC_A = 4, STREAM_ENC_E = 5, STREAM_MASK = 6 };
