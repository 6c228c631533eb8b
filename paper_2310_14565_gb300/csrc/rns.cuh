// Exact mixed-radix conversions between the residue bases Q and B.
#pragma once
#include "common.cuh"

// ---------------------------------------------------- RNS conversions
// Templated on the numbers of Q and B primes (0: read them at run time) so
// that digit arrays stay in registers; primes and constants come by value
// in the kernel parameter space (RnsArgs).

//
// PM (RnsArgs.rc.pm): every prime has folding products (PmMul) and the sizes
// are such that intermediate values need no reduction: a product is below twice
// its modulus, a digit below 4 q_i of any other prime's, so a Garner step takes
// acc + 4 q_i - v_j as it is and only the finished digits are reduced.

// Garner mixed-radix digits v of residues x (PM: below 3 p_i) over n primes
// pr[0..n), M at most; c, cs: the inverses and their companions.
template <int M, bool PM, int S>
__device__ __forceinline__ void garner(const DevPrime* pr, int n, const u64 (&c)[S][S], const u64 (&cs)[S][S],
                                       const u64* x, u64* v) {
#pragma unroll
  for (int i = 0; i < M; ++i) {
    if (i < n) {
      const DevPrime& pi = pr[i];
      u64 acc = x[i];
      if constexpr (PM) {
        const PmMul m(pi);
#pragma unroll
        for (int j = 0; j < M; ++j)
          if (j < i) acc = m.mul(acc + 4 * pi.q - v[j], c[i][j], cs[i][j]);
        if (i == 0) acc = acc >= 2 * pi.q ? acc - 2 * pi.q : acc;
        v[i] = acc >= pi.q ? acc - pi.q : acc;
      } else {
#pragma unroll
        for (int j = 0; j < M; ++j) {
          if (j < i) {
            const u64 vj = v[j] >= pi.q ? barrett64(v[j], pi) : v[j];
            acc = submod(acc, vj, pi.q);
            acc = shoup(acc, c[i][j], cs[i][j], pi.q);
          }
        }
        v[i] = acc;
      }
    }
  }
}
// ... over Q of residues x, over B of residues y
template <int K, bool PM>
__device__ __forceinline__ void garner_q(const RnsArgs& A, const u64* x, u64* v) {
  garner<K ? K : PEPSI_MAXQ, PM>(A.pr, K ? K : A.k, A.rc.cq, A.rc.cqs, x, v);
}
template <int K, int KB, bool PM>
__device__ __forceinline__ void garner_b(const RnsArgs& A, const u64* y, u64* u) {
  garner<KB ? KB : PEPSI_MAXB, PM>(A.pr + (K ? K : A.k), KB ? KB : A.kb, A.rc.cb, A.rc.cbs, y, u);
}
// true when the mixed-radix number v (n digits, M at most) exceeds h; the top
// digits decide unless they are equal
template <int M>
__device__ __forceinline__ bool digits_greater(const u64* v, const u64* h, int n) {
  bool gt = false, decided = false;
#pragma unroll
  for (int i = M - 1; i >= 0; --i) {
    if (i < n && !decided && v[i] != h[i]) {
      gt = v[i] > h[i];
      decided = true;
    }
  }
  return gt;
}
// A fixed product in the arithmetic of its prime: [0, 2q)
template <bool PM>
__device__ __forceinline__ u64 fixed_mul(u64 x, u64 w, u64 ws, const DevPrime& p) {
  if constexpr (PM)
    return PmMul(p).mul(x, w, ws);
  else
    return shoup_lazy(x, w, ws, p.q);
}
// Value of the digits v (n of them, M at most) modulo p by Horner's rule v_0 +
// r_0 (v_1 + r_1 (v_2 + ...)) with the radices r mod p: every partial value stays
// below 2 p + the largest digit, and is returned unreduced.
template <int M, bool PM>
__device__ __forceinline__ u64 horner(const u64* v, int n, const u64* r, const u64* rs, const DevPrime& p) {
  u64 acc = v[n - 1];
#pragma unroll
  for (int l = M - 2; l >= 0; --l)
    if (l < n - 1) acc = fixed_mul<PM>(acc, r[l], rs[l], p) + v[l];
  return acc;
}
// ... reduced to [0, p)
template <bool PM>
__device__ __forceinline__ u64 reduce_one(u64 x, const DevPrime& p) {
  if constexpr (PM) {
    x = PmMul(p).fold(x);
    return x >= p.q ? x - p.q : x;
  } else {
    return barrett64(x, p);
  }
}
// value of the Q-digits v (centred when neg) reduced mod B prime j
template <int K, bool PM>
__device__ __forceinline__ u64 q_digits_mod_b(const RnsArgs& A, const u64* v, bool neg, int j) {
  const int k = K ? K : A.k;
  const DevPrime& pb = A.pr[k + j];
  const u64 r = reduce_one<PM>(horner<K ? K : PEPSI_MAXQ, PM>(v, k, A.rc.qb[j], A.rc.qbs[j], pb), pb);
  return neg ? submod(r, A.rc.qmodb[j], pb.q) : r;
}
