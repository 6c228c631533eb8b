// Tensor products of ciphertexts: with their inverse transform, and summed over layers.
#include "kernels.h"
#include "ntt_block.cuh"
#include "xform.cuh"

namespace {

// a b mod q and a 128-bit sum mod q in the arithmetic of the kernel's primes
template <bool PM>
__device__ __forceinline__ u64 reduce_sum(u64 hi, u64 lo, const DevPrime& p) {
  if constexpr (PM)
    return pm_reduce(hi, lo, PmMul(p), (int)p.nbits);
  else
    return reduce128(hi, lo, p);
}
template <bool PM>
__device__ __forceinline__ u64 prod(u64 a, u64 b, const DevPrime& p) {
  if constexpr (PM)
    return pm_reduce(__umul64hi(a, b), a * b, PmMul(p), (int)p.nbits);
  else
    return mulmod(a, b, p);
}

// ------------------------------------------------------------ tensor
// Tensor product fused with its inverse transform: block per row
// (l, c, pi) of T3[L][3][k+kb][N] computes component c of the tensor of
// (A_l, B_l) at prime pi on the load of the inverse NTT, and stores the
// coefficient-form row: the tensor (a0b0, a0b1 + a1b0, a1b1) and its
// inverse NTT without a round trip of the NTT-form tensor through memory.
// Bound by the heavy multiply-add pipe (256 ciphertexts of N = 8192, k = 4: 0.56 ms).
// Its six loads beside the transforms of four ring forms spill at 64 registers: 664
// bytes compiled for folding primes alone, 788 with the other arithmetics in it.
template <bool PM, int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1)
    k_tensor_intt(DevView V, const u64* __restrict__ AQ, const u64* __restrict__ AB, const u64* __restrict__ BQ,
                  const u64* __restrict__ BB, const u64* __restrict__ cstQ, const u64* __restrict__ side,
                  u64* __restrict__ T3, int square) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k, kb = V.kb, np = k + kb;
  const size_t r = blockIdx.x;
  const int pi = (int)(r % np);
  const size_t o = r / np;  // l * 3 + c
  const int c = (int)(o % 3);
  const size_t l = o / 3;
  const DevPrime pr = V.pr[pi];
  const u64 *A, *Bp;
  size_t o0, o1;
  u64 cb = 0;  // constant added to b0 (NTT form: the same at every point)
  if (pi < k) {
    A = AQ;
    Bp = BQ;
    o0 = ((l * 2 + 0) * k + pi) * N;
    o1 = ((l * 2 + 1) * k + pi) * N;
    if (!square && cstQ) cb = cstQ[pi];
  } else {
    A = AB;
    Bp = BB;
    o0 = ((l * 2 + 0) * kb + (pi - k)) * N;
    o1 = ((l * 2 + 1) * kb + (pi - k)) * N;
    if (!square && side) cb = side[l * kb + (pi - k)];
  }
  const u64* a0 = A + o0;
  const u64* a1 = A + o1;
  const u64* b0 = Bp + o0;
  const u64* b1 = Bp + o1;
  const RowSt st(T3 + r * N);
  if (square) {
    if (c == 0)
      ntt_inv_gg<PM, RING>(sm, [&](int x) { return prod<PM>(a0[x], a0[x], pr); }, st, V, pi);
    else if (c == 1)
      ntt_inv_gg<PM, RING>(
          sm,
          [&](int x) {
            const u64 m = prod<PM>(a0[x], a1[x], pr);
            return addmod(m, m, pr.q);
          },
          st, V, pi);
    else
      ntt_inv_gg<PM, RING>(sm, [&](int x) { return prod<PM>(a1[x], a1[x], pr); }, st, V, pi);
  } else {
    if (c == 0)
      ntt_inv_gg<PM, RING>(sm, [&](int x) { return prod<PM>(a0[x], addmod(b0[x], cb, pr.q), pr); }, st, V, pi);
    else if (c == 1)
      ntt_inv_gg<PM, RING>(
          sm,
          [&](int x) {
            u64 lo = 0, hi = 0;
            mac128(lo, hi, a0[x], b1[x]);
            mac128(lo, hi, a1[x], addmod(b0[x], cb, pr.q));
            return reduce_sum<PM>(hi, lo, pr);
          },
          st, V, pi);
    else
      ntt_inv_gg<PM, RING>(sm, [&](int x) { return prod<PM>(a1[x], b1[x], pr); }, st, V, pi);
  }
}

// Lazy rescaling: X[c][pi][n] (+)= sum over layers l < L of component c of
// the tensor of (A_l, B_l), in NTT form over Q u B, each layer's tensor
// times its value plaintext VP[l][pi][n] when VP is given (labelled PSI /
// PSI-Sum).  The products of each (prime, point) are summed in 128 bits
// and reduced once per 16 layers (at most 32 products below 2^122 each
// stay below 2^127), so the sum is exact mod every prime; the integer it
// represents is the sum of the layers' exact integer tensors (times the
// values) as long as B holds it (sized at setup).
// Four blocks per SM (64 registers a thread, a few spilled): at the paper
// shape the sums of two 263-layer chunks took 0.27 ms against 0.31 ms with
// three blocks (80 registers), whose 1152 blocks left a half-empty last wave.
constexpr int TS_PTS = 64, TS_SLICES = 4;
__global__ void __launch_bounds__(TS_PTS * TS_SLICES, 4) k_tensor_sum(DevView V, const u64* __restrict__ AQ, const u64* __restrict__ AB,
                             const u64* __restrict__ BQ, const u64* __restrict__ BB, const u64* __restrict__ cstQ,
                             const u64* __restrict__ side, const u64* __restrict__ VP, u64* __restrict__ X, int L,
                             int square, int init) {
  // block: TS_PTS consecutive (prime, point) words x TS_SLICES slices of
  // the layers; each slice sums every TS_SLICES-th layer, and the slices'
  // residues are added at the end
  __shared__ u64 part[3][TS_SLICES][TS_PTS];
  const int N = V.N, k = V.k, kb = V.kb, np = k + kb;
  const int tp = threadIdx.x % TS_PTS, slice = threadIdx.x / TS_PTS;
  const size_t idx = (size_t)blockIdx.x * TS_PTS + tp;  // over np*N
  const bool active = idx < (size_t)np * N;  // every thread reaches the barrier below
  const int n = active ? (int)(idx % N) : 0;
  const int pi = active ? (int)(idx / N) : 0;
  const DevPrime pr = V.pr[pi];
  const bool inQ = pi < k;
  const int kk = inQ ? k : kb, pp = inQ ? pi : pi - k;
  const u64* A = inQ ? AQ : AB;
  const u64* Bp = inQ ? BQ : BB;
  const u64 cq = (inQ && cstQ) ? cstQ[pi] : 0;
  const size_t cs = (size_t)kk * N;  // component stride of the operands
  const PmMul pm(pr);
  auto reduce = [&](u64 hi, u64 lo) { return pr.pm ? pm_reduce(hi, lo, pm, (int)pr.nbits) : reduce128(hi, lo, pr); };
  u64 s0l = 0, s0h = 0, s1l = 0, s1h = 0, s2l = 0, s2h = 0;
  int cnt = 0;
  for (int l = active ? slice : L; l < L; l += TS_SLICES) {
    const size_t o0 = ((size_t)l * 2 * kk + pp) * N + n;
    const u64 a0 = A[o0], a1 = A[o0 + cs];
    u64 b0 = a0, b1 = a1;
    if (!square) {
      b0 = Bp[o0];
      b1 = Bp[o0 + cs];
      if (inQ) {
        b0 = addmod(b0, cq, pr.q);
      } else if (side) {
        b0 = addmod(b0, side[(size_t)l * kb + pp], pr.q);
      }
    }
    if (VP) {
      const u64 v = VP[((size_t)l * np + pi) * N + n];
      u64 lo = 0, hi = 0;
      mac128(lo, hi, a0, b1);
      mac128(lo, hi, a1, b0);
      mac128(s0l, s0h, mulmod(a0, b0, pr), v);
      mac128(s1l, s1h, reduce128(hi, lo, pr), v);
      mac128(s2l, s2h, mulmod(a1, b1, pr), v);
    } else {
      mac128(s0l, s0h, a0, b0);
      mac128(s1l, s1h, a0, b1);
      mac128(s1l, s1h, a1, b0);
      mac128(s2l, s2h, a1, b1);
    }
    if ((++cnt & 15) == 0) {
      s0l = reduce(s0h, s0l);
      s1l = reduce(s1h, s1l);
      s2l = reduce(s2h, s2l);
      s0h = s1h = s2h = 0;
    }
  }
  part[0][slice][tp] = reduce(s0h, s0l);
  part[1][slice][tp] = reduce(s1h, s1l);
  part[2][slice][tp] = reduce(s2h, s2l);
  __syncthreads();
  if (slice == 0 && active) {
    u64* o = X + (size_t)pi * N + n;
    const size_t os = (size_t)np * N;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u64 d = part[c][0][tp];
#pragma unroll
      for (int sl = 1; sl < TS_SLICES; ++sl) d = addmod(d, part[c][sl][tp], pr.q);
      o[c * os] = init ? d : addmod(d, o[c * os], pr.q);
    }
  }
}

}  // namespace

void launch_tensor_intt(const DevView& V, const u64* AQ, const u64* AB, const u64* BQ, const u64* BB,
                        const u64* cstQ, const u64* side, u64* T3, int L, bool square, cudaStream_t st) {
  const size_t rows = (size_t)L * 3 * (V.k + V.kb);
  if (!rows) return;
  auto go = [&](auto kernel) {
    kernel<<<(unsigned)rows, xform_threads(V, rows), (size_t)V.N * 8, st>>>(V, AQ, AB, BQ, BB, cstQ, side, T3,
                                                                          square ? 1 : 0);
  };
  in_form(V, [&](auto pm, auto ring) { go(k_tensor_intt<decltype(pm)::value, decltype(ring)::value>); });
}

void launch_tensor_sum(const DevView& V, const u64* AQ, const u64* AB, const u64* BQ, const u64* BB,
                       const u64* cstQ, const u64* side, const u64* VP, u64* X, int L, bool square, bool init,
                       cudaStream_t st) {
  const size_t total = (size_t)(V.k + V.kb) * V.N;
  k_tensor_sum<<<(unsigned)((total + TS_PTS - 1) / TS_PTS), TS_PTS * TS_SLICES, 0, st>>>(V, AQ, AB, BQ, BB, cstQ, side, VP, X, L,
                                                                          square ? 1 : 0, init ? 1 : 0);
}

cudaError_t tensor_init() {
  return allow_smem({(const void*)k_tensor_intt<true, RING_ANY>, (const void*)k_tensor_intt<false, RING_ANY>});
}
