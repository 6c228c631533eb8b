// Block-cooperative negacyclic NTT on a shared-memory polynomial.
//
// Forward: natural-order coefficients in, values at psi^(2 brev(i)+1) in
// position i out (radix-2 Cooley-Tukey with twiddles psi^brev(m+i), the
// merged negacyclic form of Longa-Naehrig), Harvey's lazy butterflies.
// Inverse: Gentleman-Sande with psi^-brev(m+i), then the factor N^-1.
//
// The log2 N radix-2 stages run in phases of RR <= 3 consecutive stages.  The
// butterflies of stages [s0, s0+RR) only combine the 2^RR elements base + i * (N >> (s0+RR)), i < 2^RR, so a thread loads such a
// group into registers, runs the RR stages there and stores it back: one
// shared-memory round trip and one barrier per phase instead of per stage.
// Every thread of the block must call these (they contain __syncthreads);
// any block size works (threads loop over the groups).
//
// Shared-memory layout: logical element x lives at word nsw(x) = x ^ ((x >> 4)
// & 15).  Groups of a phase are read at element strides 2^k; with the XOR of
// the higher index bits into the low four, the 16 words a half-warp reads
// fall into 16 different 8-byte bank pairs for every such stride, and runs
// of consecutive elements stay conflict-free.  Callers filling or reading
// the array index it through nsw().
#pragma once
#include <type_traits>
#include "common.cuh"

__host__ __device__ __forceinline__ constexpr int nsw(int x) { return x ^ ((x >> 4) & 15); }

// Element base + c of the array for base and c with no common bit, from nb =
// nsw(base) * sizeof(T).  nsw is linear over XOR, so only c's part of the low four
// bits is XORed in and the rest is an offset: with c a constant (the phases of
// the fixed ring sizes) that is one operation or none per access, instead of the
// five of nsw(base + c) on the ALU pipe, which the transforms keep as busy as the
// multiply-add pipe.
template <class T>
__device__ __forceinline__ T& at(T* a, u32 nb, int c) {
  const int low = (c & 15) ^ ((c >> 4) & 15), high = c & ~15;
  return *reinterpret_cast<T*>(reinterpret_cast<char*>(a) + (nb ^ (u32)(low * (int)sizeof(T))) + high * (int)sizeof(T));
}

// The same where c is not a constant: nsw of the sum is the shorter form.
template <bool FIXED, class T>
__device__ __forceinline__ T& at_phase(T* a, int base, u32 nb, int c) {
  if constexpr (FIXED)
    return at(a, nb, c);
  else
    return a[nsw(base + c)];
}

namespace nttd {

// Arithmetic of a transform's modulus.  mul(x, t) multiplies by a table entry
// t = (w, companion) into [0, 2q).
//  - Shoup<G>: any q below 2^61.  G (q < 2^59): the forward butterfly's sum input
//    is not reduced below 2q first, so values grow by 2q a stage (the product
//    takes any 64-bit input): from [0, 4q) they stay below (4 + 2 log2 N) q <=
//    32 q, which fits 64 bits, and one Barrett reduction at the end reduces them.
//  - Pm: q = 2^n - d, n <= 57 (PmMul, inputs below 2^(n+5)): forward as above; the
//    inverse's sums double from 4q to at most 32q over the three stages of a
//    phase, and a fold of the sums at its end brings them below 2q.
//  - Small: 32-bit words for a modulus below 2^30 (the plaintext modulus t), where
//    Shoup's product takes one 32x32 high product and two low ones; the upper half
//    of a Shoup companion floor(w 2^64 / q) is floor(w 2^32 / q).
template <bool G>
struct Shoup {
  typedef u64 T;
  static constexpr bool kGrow = G, kPm = false;
  u64 q, m64;
  __device__ __forceinline__ explicit Shoup(const DevPrime& p) : q(p.q), m64(p.m64) {}
  __device__ __forceinline__ u64 mul(u64 x, const ulonglong2& t) const { return shoup_lazy(x, t.x, t.y, q); }
};
struct Pm {
  typedef u64 T;
  static constexpr bool kGrow = true, kPm = true;
  PmMul m;
  u64 q;
  __device__ __forceinline__ explicit Pm(const DevPrime& p) : m(p), q(p.q) {}
  __device__ __forceinline__ u64 mul(u64 x, const ulonglong2& t) const { return m.mul(x, t.x, t.y); }
};
struct Small {
  typedef u32 T;
  static constexpr bool kGrow = false, kPm = false;
  u32 q;
  __device__ __forceinline__ explicit Small(const DevPrime& p) : q((u32)p.q) {}
  __device__ __forceinline__ u32 mul(u32 x, const ulonglong2& t) const {
    return x * (u32)t.x - __umulhi(x, (u32)(t.y >> 32)) * q;
  }
};

// Forward stages [s0, s0 + RR) on one group of 2^RR elements held in
// registers, element i of the group at base + i * 2^(logN - s0 - RR).
// Twiddles come as (w, companion) pairs, one 16-byte load each.
template <int RR, class A>
__device__ __forceinline__ void fwd_group(u64 (&x)[1 << RR], int base, int logN, int s0, const A& ar,
                                          const ulonglong2* __restrict__ tw) {
  constexpr int E = 1 << RR;
  const u64 q2 = 2 * ar.q;
#pragma unroll
  for (int ss = 0; ss < RR; ++ss) {
    const int s = s0 + ss;
    const int half = 1 << (RR - 1 - ss);
    // base has zero bits where i * stride lands, so the twiddle index of
    // butterfly i splits into a group part and i >> (RR - ss): stage ss of
    // the phase needs only 2^ss distinct twiddles
    const int tbase = (1 << s) + (base >> (logN - s));
    ulonglong2 Wt[1 << (RR - 1)];
#pragma unroll
    for (int d = 0; d < (1 << ss); ++d) Wt[d] = __ldg(tw + tbase + d);
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if ((i & half) == 0) {
        u64 U = x[i];
        if constexpr (!A::kGrow) U = U >= q2 ? U - q2 : U;
        const u64 T = ar.mul(x[i + half], Wt[i >> (RR - ss)]);
        x[i] = U + T;
        x[i + half] = U + q2 - T;
      }
    }
  }
}
// The transform's end: [0, 4q), or the grown range, -> [0, q)
template <int E, class A>
__device__ __forceinline__ void fwd_final(u64 (&x)[E], const A& ar) {
  const u64 q = ar.q, q2 = 2 * q;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    u64 v = x[i];
    if constexpr (A::kPm) {
      v = ar.m.fold(v);
    } else if constexpr (A::kGrow) {
      v -= __umul64hi(v, ar.m64) * q;  // floor(v m64 / 2^64) is short of floor(v / q) by at most 1
    } else {
      v = v >= q2 ? v - q2 : v;
    }
    x[i] = v >= q ? v - q : v;
  }
}
// Inverse (Gentleman-Sande) stages s0 + RR - 1 down to LO (the first LO of
// the phase are left out) on one group.  Shoup: values stay in [0, 2q).  Pm:
// sums double from [0, 4q) a stage.
template <int RR, int LO, class A>
__device__ __forceinline__ void inv_stages(typename A::T (&x)[1 << RR], int base, int logN, int s0, const A& ar,
                                           const ulonglong2* __restrict__ itw) {
  typedef typename A::T T;
  constexpr int E = 1 << RR;
  const T q2 = 2 * ar.q;
#pragma unroll
  for (int ss = RR - 1; ss >= LO; --ss) {
    const int s = s0 + ss;
    const int half = 1 << (RR - 1 - ss);
    const int tbase = (1 << s) + (base >> (logN - s));
    const T c = A::kPm ? (2 * q2) << (RR - 1 - ss) : q2;  // bound of V
    ulonglong2 Wt[1 << (RR - 1)];
#pragma unroll
    for (int d = 0; d < (1 << ss); ++d) Wt[d] = __ldg(itw + tbase + d);
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if ((i & half) == 0) {
        const T U = x[i], V = x[i + half];
        T S = U + V;
        if constexpr (!A::kPm) S = S >= q2 ? S - q2 : S;
        x[i] = S;
        x[i + half] = ar.mul((T)(U + c - V), Wt[i >> (RR - ss)]);
      }
    }
  }
}
// A whole phase; Pm: the last stage's sums are folded below 2q.
template <int RR, class A>
__device__ __forceinline__ void inv_group(typename A::T (&x)[1 << RR], int base, int logN, int s0, const A& ar,
                                          const ulonglong2* __restrict__ itw) {
  inv_stages<RR, 0>(x, base, logN, s0, ar, itw);
  if constexpr (A::kPm) {
#pragma unroll
    for (int i = 0; i < (1 << RR) / 2; ++i) x[i] = ar.m.fold(x[i]);
  }
}
// times N^-1, [0, 2q) -> [0, q)
template <int E, class A>
__device__ __forceinline__ void inv_final(typename A::T (&x)[E], const A& ar, const ulonglong2& ninv) {
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const typename A::T v = ar.mul(x[i], ninv);
    x[i] = v >= ar.q ? v - ar.q : v;
  }
}

// Stages 2, 1, 0 of the inverse on the radix-8 group at base, with the
// factor N^-1: the sums of stage 0 are multiplied by N^-1, the differences
// by the table's entry 0 (the stage-0 twiddle times N^-1) instead of by the
// twiddle, then every element is reduced to [0, q).  The same residues as
// inv_group<3> at s0 = 0 followed by inv_final, with half the products of
// the final scaling.
template <class A>
__device__ __forceinline__ void inv_group_last(typename A::T (&x)[8], int base, int logN, const A& ar,
                                               const ulonglong2* __restrict__ itw, const ulonglong2& ninv) {
  typedef typename A::T T;
  inv_stages<3, 1>(x, base, logN, 0, ar, itw);
  const T q = ar.q, q2 = 2 * q, c = A::kPm ? 8 * q2 : q2;
  const ulonglong2 wn = __ldg(itw);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const T U = x[i], V = x[i + 4];
    T S = U + V;
    if constexpr (!A::kPm) S = S >= q2 ? S - q2 : S;
    const T a = ar.mul(S, ninv), b = ar.mul((T)(U + c - V), wn);
    x[i] = a >= q ? a - q : a;
    x[i + 4] = b >= q ? b - q : b;
  }
}

// FIXED: N, logN and s0 are constants of the instance (at_phase).
template <int RR, bool FIXED, class A>
__device__ __forceinline__ void fwd_phase(u64* a, int N, int logN, int s0, const A& ar,
                                          const ulonglong2* __restrict__ tw, bool last) {
  constexpr int E = 1 << RR;
  const int slog = logN - s0 - RR;  // log2 of the element stride inside a group
  const int groups = N >> RR;
  for (int g = threadIdx.x; g < groups; g += blockDim.x) {
    const int base = ((g >> slog) << (slog + RR)) + (g & ((1 << slog) - 1));
    const u32 nb = (u32)nsw(base) * 8;
    u64 x[E];
#pragma unroll
    for (int i = 0; i < E; ++i) x[i] = at_phase<FIXED>(a, base, nb, i << slog);
    fwd_group<RR>(x, base, logN, s0, ar, tw);
    if (last) fwd_final<E>(x, ar);
#pragma unroll
    for (int i = 0; i < E; ++i) at_phase<FIXED>(a, base, nb, i << slog) = x[i];
  }
}

template <int RR, bool FIXED, class A>
__device__ __forceinline__ void inv_phase(typename A::T* a, int N, int logN, int s0, const A& ar,
                                          const ulonglong2* __restrict__ itw, bool last, const ulonglong2& ninv) {
  typedef typename A::T T;
  constexpr int E = 1 << RR;
  const int slog = logN - s0 - RR;
  const int groups = N >> RR;
  for (int g = threadIdx.x; g < groups; g += blockDim.x) {
    const int base = ((g >> slog) << (slog + RR)) + (g & ((1 << slog) - 1));
    const u32 nb = (u32)nsw(base) * (u32)sizeof(T);
    T x[E];
#pragma unroll
    for (int i = 0; i < E; ++i) x[i] = at_phase<FIXED>(a, base, nb, i << slog);
    inv_group<RR>(x, base, logN, s0, ar, itw);
    if (last) inv_final<E>(x, ar, ninv);
#pragma unroll
    for (int i = 0; i < E; ++i) at_phase<FIXED>(a, base, nb, i << slog) = x[i];
  }
}

}  // namespace nttd

// a[0..N) in [0, 4q) on entry, [0, q) on exit.  Phases of three stages
// from stage 0, then the remaining one or two.
template <class A>
__device__ __forceinline__ void ntt_fwd_block(u64* a, int N, int logN, const A& ar, const ulonglong2* __restrict__ tw) {
  int s0 = 0;
  for (; s0 + 3 <= logN; s0 += 3) {
    nttd::fwd_phase<3, false>(a, N, logN, s0, ar, tw, s0 + 3 == logN);
    __syncthreads();
  }
  const int rem = logN - s0;
  if (rem == 2) nttd::fwd_phase<2, false>(a, N, logN, s0, ar, tw, true);
  if (rem == 1) nttd::fwd_phase<1, false>(a, N, logN, s0, ar, tw, true);
  if (rem) __syncthreads();
}

// a[0..N) in [0, 2q) on entry, [0, q) on exit.  The forward phases in
// reverse order: the remainder first, then three stages at a time.
template <class A>
__device__ __forceinline__ void ntt_inv_block(typename A::T* a, int N, int logN, const A& ar,
                                              const ulonglong2* __restrict__ itw, const ulonglong2& ninv) {
  const int rem = logN % 3;
  int s0 = logN - rem;
  if (rem == 2) nttd::inv_phase<2, false>(a, N, logN, s0, ar, itw, s0 == 0, ninv);
  if (rem == 1) nttd::inv_phase<1, false>(a, N, logN, s0, ar, itw, s0 == 0, ninv);
  if (rem) __syncthreads();
  for (s0 -= 3; s0 >= 0; s0 -= 3) {
    nttd::inv_phase<3, false>(a, N, logN, s0, ar, itw, s0 == 0, ninv);
    __syncthreads();
  }
}

__device__ __forceinline__ void ntt_fwd_view(u64* a, const DevView& V, int pi) {
  const DevPrime P = V.pr[pi];
  const ulonglong2* tw = V.twp + (size_t)pi * V.N;
  if (P.pm)
    ntt_fwd_block(a, V.N, V.logN, nttd::Pm(P), tw);
  else
    ntt_fwd_block(a, V.N, V.logN, nttd::Shoup<false>(P), tw);
}
__device__ __forceinline__ void ntt_inv_view(u64* a, const DevView& V, int pi) {
  const DevPrime P = V.pr[pi];
  const ulonglong2* itw = V.itwp + (size_t)pi * V.N;
  const ulonglong2 ninv = make_ulonglong2(P.ninv, P.ninvs);
  if (P.pm)
    ntt_inv_block(a, V.N, V.logN, nttd::Pm(P), itw, ninv);
  else
    ntt_inv_block(a, V.N, V.logN, nttd::Shoup<false>(P), itw, ninv);
}

// Row accessors for the global-to-global transforms.  A functor with a
// pair(x, ...) member moves elements x and x + 1 (x even) together; the
// transforms use it for the groups of consecutive elements (the first group
// of the inverse, the last of the forward).  The row accessors do one
// 16-byte access when the row is 16-byte aligned (rows are whole multiples
// of N words from their base, so the test is uniform over a block) and two
// 8-byte accesses otherwise: caller buffers need only 8-byte alignment.
// Plain lambdas are used element by element.
template <class T, class = void>
struct has_pair : std::false_type {};
template <class T>
struct has_pair<T, std::void_t<decltype(&T::pair)>> : std::true_type {};
__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
struct RowLd {
  const u64* p;
  bool v16;
  __device__ __forceinline__ explicit RowLd(const u64* row) : p(row), v16(aligned16(row)) {}
  __device__ __forceinline__ u64 operator()(int x) const { return p[x]; }
  __device__ __forceinline__ void pair(int x, u64& a, u64& b) const {
    if (v16) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(p + x);
      a = w.x;
      b = w.y;
    } else {
      a = p[x];
      b = p[x + 1];
    }
  }
};
struct RowSt {
  u64* p;
  bool v16;
  __device__ __forceinline__ explicit RowSt(u64* row) : p(row), v16(aligned16(row)) {}
  __device__ __forceinline__ void operator()(int x, u64 v) const { p[x] = v; }
  __device__ __forceinline__ void pair(int x, u64 a, u64 b) const {
    if (v16) {
      *reinterpret_cast<ulonglong2*>(p + x) = make_ulonglong2(a, b);
    } else {
      p[x] = a;
      p[x + 1] = b;
    }
  }
};
// the split operand format of the multiply-accumulate (shift s)
struct SplitSt {
  RowSt r;
  u64 s;
  __device__ __forceinline__ SplitSt(u64* row, u64 shift) : r(row), s(shift) {}
  __device__ __forceinline__ void operator()(int x, u64 v) const { r(x, to_split(v, s)); }
  __device__ __forceinline__ void pair(int x, u64 a, u64 b) const { r.pair(x, to_split(a, s), to_split(b, s)); }
};
// the split operand format plus the 32-bit sum of each word's halves
struct SplitSumSt {
  SplitSt w;
  u32* sum;
  __device__ __forceinline__ SplitSumSt(u64* row, u32* sums, u64 shift) : w(row, shift), sum(sums) {}
  __device__ __forceinline__ static u32 halves(u64 v) { return (u32)v + (u32)(v >> 32); }
  __device__ __forceinline__ void operator()(int x, u64 v) const {
    const u64 t = to_split(v, w.s);
    w.r(x, t);
    sum[x] = halves(t);
  }
  __device__ __forceinline__ void pair(int x, u64 a, u64 b) const {
    const u64 ta = to_split(a, w.s), tb = to_split(b, w.s);
    w.r.pair(x, ta, tb);
    sum[x] = halves(ta);
    sum[x + 1] = halves(tb);
  }
};
template <int E, class T, class Load>
__device__ __forceinline__ void load_run(T (&x)[E], const Load& ld, int base) {
  if constexpr (has_pair<Load>::value && E >= 2) {
#pragma unroll
    for (int i = 0; i < E; i += 2) ld.pair(base + i, x[i], x[i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i) x[i] = ld(base + i);
  }
}
template <int E, class Store>
__device__ __forceinline__ void store_run(const u64 (&x)[E], const Store& st, int base) {
  if constexpr (has_pair<Store>::value && E >= 2) {
#pragma unroll
    for (int i = 0; i < E; i += 2) st.pair(base + i, x[i], x[i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i) st(base + i, x[i]);
  }
}

// Transforms from a row in global memory to a row in global memory through
// the shared-memory array a[].  The first three stages run on the registers
// of the global load and the last R stages (R = 1, 2 or 3, the rest after
// radix-8 phases) on those of the global store, so of the log2(N) stages
// only the middle ones take shared-memory phases (N = 8192: three instead
// of five).  The butterflies are those of ntt_fwd_block / ntt_inv_block, so
// are the results.  ld(x) returns input element x (forward:
// in [0, 4q); inverse: in [0, 2q)); st(x, v) receives output element x,
// reduced.  Every read through ld comes before a barrier of the whole block
// that every st comes after, so input and output rows may alias.  Every
// thread of the block must call these.
// Only the exchange around stages 0-2 crosses the whole block.  After stage 2
// the transform falls into 8 parts of N/8 elements, each the work of N/64
// consecutive threads, which one named barrier joins; after stage 5 the parts
// of N/64 elements lie within a warp's 256 elements, and the short last (first)
// phase keeps to the warp's own elements too, so warp barriers do and the warps
// of a block drift apart and fill both the multiply-add and the ALU pipe.
template <int LOGN>
__device__ __forceinline__ void part_sync() {
  constexpr int T = 1 << (LOGN - 6);
  const int sets = (int)blockDim.x / T;
  if (sets > 1 && sets <= 15)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / T), "n"(T) : "memory");
  else
    __syncthreads();
}
template <int LOGN, class A, class Load, class Store>
__device__ __forceinline__ void ntt_fwd_fused(u64* a, const Load& ld, const Store& st, const A& ar,
                                              const ulonglong2* __restrict__ tw) {
  constexpr int N = 1 << LOGN, R = (LOGN - 4) % 3 + 1, M = (LOGN - 3 - R) / 3, S8 = LOGN - 3;
  for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x) {  // stages 0-2
    u64 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = ld(g + (i << S8));
    nttd::fwd_group<3>(x, g, LOGN, 0, ar, tw);
    const u32 nb = (u32)nsw(g) * 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) at(a, nb, i << S8) = x[i];
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < M; ++m) {
    nttd::fwd_phase<3, true>(a, N, LOGN, 3 + 3 * m, ar, tw, false);
    if (m == 0)
      part_sync<LOGN>();
    else
      __syncwarp();
  }
  for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x) {  // stages LOGN-R .. LOGN-1 of the warp's 256 elements
#pragma unroll
    for (int it = 0; it < (8 >> R); ++it) {
      const int base = (((g & ~31) << 3) + ((it * 32 + (g & 31)) << R));
      const u32 nb = (u32)nsw(base) * 8;
      u64 x[1 << R];
#pragma unroll
      for (int i = 0; i < (1 << R); ++i) x[i] = at(a, nb, i);
      nttd::fwd_group<R>(x, base, LOGN, LOGN - R, ar, tw);
      nttd::fwd_final<1 << R>(x, ar);
      store_run<1 << R>(x, st, base);
    }
  }
}
template <int LOGN, class A, class Load, class Store>
__device__ __forceinline__ void ntt_inv_fused(typename A::T* a, const Load& ld, const Store& st, const A& ar,
                                              const ulonglong2* __restrict__ itw, const ulonglong2& ninv) {
  typedef typename A::T T;
  constexpr int N = 1 << LOGN, R = (LOGN - 4) % 3 + 1, M = (LOGN - 3 - R) / 3, S8 = LOGN - 3;
  for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x) {  // stages LOGN-1 .. LOGN-R of the warp's 256 elements
#pragma unroll
    for (int it = 0; it < (8 >> R); ++it) {
      const int base = (((g & ~31) << 3) + ((it * 32 + (g & 31)) << R));
      T x[1 << R];
      load_run<1 << R>(x, ld, base);
      nttd::inv_group<R>(x, base, LOGN, LOGN - R, ar, itw);
      const u32 nb = (u32)nsw(base) * (u32)sizeof(T);
#pragma unroll
      for (int i = 0; i < (1 << R); ++i) at(a, nb, i) = x[i];
    }
  }
  __syncwarp();
#pragma unroll
  for (int m = M - 1; m >= 0; --m) {
    nttd::inv_phase<3, true>(a, N, LOGN, 3 + 3 * m, ar, itw, false, ninv);
    if (m > 1)
      __syncwarp();
    else if (m == 1)
      part_sync<LOGN>();
    else
      __syncthreads();
  }
  for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x) {  // stages 2-0 and N^-1
    const u32 nb = (u32)nsw(g) * (u32)sizeof(T);
    T x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = at(a, nb, i << S8);
    nttd::inv_group_last(x, g, LOGN, ar, itw, ninv);
#pragma unroll
    for (int i = 0; i < 8; ++i) st(g + (i << S8), x[i]);
  }
}

// Global-to-global transforms of row pi with the fused forms for the ring
// sizes of the workloads (N = 4096, 8192, 16384), else load, block
// transform and store; each in the arithmetic of the row's prime.
template <int RING, class A, class Load, class Store>
__device__ __forceinline__ void ntt_fwd_with(u64* a, const Load& ld, const Store& st, const A& ar, int N, int logN,
                                             const ulonglong2* __restrict__ tw) {
  if constexpr (RING != RING_SMALL) {
    switch (logN) {
      case 12: ntt_fwd_fused<12>(a, ld, st, ar, tw); return;
      case 13: ntt_fwd_fused<13>(a, ld, st, ar, tw); return;
      case 14: ntt_fwd_fused<14>(a, ld, st, ar, tw); return;
      default: break;
    }
  }
  for (int x = threadIdx.x; x < N; x += blockDim.x) a[nsw(x)] = ld(x);
  __syncthreads();
  ntt_fwd_block(a, N, logN, ar, tw);
  for (int x = threadIdx.x; x < N; x += blockDim.x) st(x, a[nsw(x)]);
}
template <int RING, class A, class Load, class Store>
__device__ __forceinline__ void ntt_inv_with(typename A::T* a, const Load& ld, const Store& st, const A& ar, int N,
                                             int logN, const ulonglong2* __restrict__ itw, const ulonglong2& ninv) {
  if constexpr (RING != RING_SMALL) {
    switch (logN) {
      case 12: ntt_inv_fused<12>(a, ld, st, ar, itw, ninv); return;
      case 13: ntt_inv_fused<13>(a, ld, st, ar, itw, ninv); return;
      case 14: ntt_inv_fused<14>(a, ld, st, ar, itw, ninv); return;
      default: break;
    }
  }
  for (int x = threadIdx.x; x < N; x += blockDim.x) a[nsw(x)] = ld(x);
  __syncthreads();
  ntt_inv_block(a, N, logN, ar, itw, ninv);
  for (int x = threadIdx.x; x < N; x += blockDim.x) st(x, a[nsw(x)]);
}
// PM: every prime the kernel meets has folding products (DevView::allpm).  The
// kernels come in both forms: with the other arithmetics compiled in beside it,
// the compiler moved so much out of the branches that the inverse kernels spilled
// more (k_tensor_intt 788 bytes against 664, k_relin_axpy_intt 400 against 332,
// k_axpy_intt 136 against 72); 1200 x 4 rows of N = 8192 forward 281 -> 269 us, the
// products of 256 ciphertexts 2.39 -> 2.33 ms.
template <bool PM = false, int RING = RING_ANY, class Load, class Store>
__device__ __forceinline__ void ntt_fwd_gg(u64* a, const Load& ld, const Store& st, const DevView& V, int pi) {
  const ulonglong2* tw = V.twp + (size_t)pi * V.N;
  const DevPrime P = V.pr[pi];
  if constexpr (PM)
    ntt_fwd_with<RING>(a, ld, st, nttd::Pm(P), V.N, V.logN, tw);
  else if (P.pm)
    ntt_fwd_with<RING>(a, ld, st, nttd::Pm(P), V.N, V.logN, tw);
  else if (P.q < (1ull << 59))
    ntt_fwd_with<RING>(a, ld, st, nttd::Shoup<true>(P), V.N, V.logN, tw);
  else
    ntt_fwd_with<RING>(a, ld, st, nttd::Shoup<false>(P), V.N, V.logN, tw);
}
template <bool PM = false, int RING = RING_ANY, class Load, class Store>
__device__ __forceinline__ void ntt_inv_gg(u64* a, const Load& ld, const Store& st, const DevView& V, int pi) {
  const ulonglong2* itw = V.itwp + (size_t)pi * V.N;
  const DevPrime P = V.pr[pi];
  const ulonglong2 ninv = make_ulonglong2(P.ninv, P.ninvs);
  if constexpr (PM)
    ntt_inv_with<RING>(a, ld, st, nttd::Pm(P), V.N, V.logN, itw, ninv);
  else if (P.pm)
    ntt_inv_with<RING>(a, ld, st, nttd::Pm(P), V.N, V.logN, itw, ninv);
  else
    ntt_inv_with<RING>(a, ld, st, nttd::Shoup<false>(P), V.N, V.logN, itw, ninv);
}

// ntt_inv_gg for a modulus q_pi below 2^30 (the plaintext modulus) in 32-bit
// words: a[] holds N 32-bit words, ld(x) returns element x in [0, 2q) as
// u32, st(x, v) receives it reduced.  The same residues as ntt_inv_gg.
template <int RING = RING_ANY, class Load, class Store>
__device__ __forceinline__ void ntt_inv_gg_small(u32* a, const Load& ld, const Store& st, const DevView& V, int pi) {
  const DevPrime P = V.pr[pi];
  ntt_inv_with<RING>(a, ld, st, nttd::Small(P), V.N, V.logN, V.itwp + (size_t)pi * V.N, make_ulonglong2(P.ninv, P.ninvs));
}
