// Base extension and exact rounding.
#include "kernels.h"
#include "rns.cuh"
#include "xform.cuh"

namespace {

// side[layer][j]: the lift of (x + cst) mod Q less the lift of x, mod p_j, at
// coefficient 0 of component 0.
template <int K, int KB, bool PM>
__device__ __forceinline__ void lift_side(const RnsArgs& A, const u64* __restrict__ src, int layer,
                                          const u64* __restrict__ cst, u64* side) {
  constexpr int MQ = K ? K : PEPSI_MAXQ;
  const int N = A.N, k = K ? K : A.k, kb = KB ? KB : A.kb;
#pragma unroll 1
  for (int plain = 0; plain < 2; ++plain) {
    u64 x[MQ], v[MQ];
#pragma unroll
    for (int i = 0; i < MQ; ++i)
      if (K || i < k) {
        x[i] = src[((size_t)layer * 2 * k + i) * N];
        if (!plain) x[i] = addmod(x[i], cst[i], A.pr[i].q);
      }
    garner_q<K, PM>(A, x, v);
    const bool neg = digits_greater<MQ>(v, A.rc.qhalf_dig, k);
#pragma unroll 1
    for (int j = 0; j < kb; ++j) {
      const u64 w = q_digits_mod_b<K, PM>(A, v, neg, j);
      u64& s = side[(size_t)layer * kb + j];
      s = plain ? submod(s, w, A.pr[k + j].q) : w;
    }
  }
}
// Q -> B extension, thread per coefficient; the first `ns` blocks, a thread per
// layer, make side[] beside the others (in a launch of its own it cost small
// evaluations 4 to 10 us a lift; in every thread of coefficient 0 its second set of
// digits cost registers, 232 at k = kb = 8).  The run-time generic form keeps ns = 0
// and k_lift_side: with both loops it took 200 registers instead of 34.
template <int K, int KB, bool PM>
__global__ void __launch_bounds__(128, K == 0 ? 1 : K < 8 ? 16 : 12) k_lift(const __grid_constant__ RnsArgs A, const u64* __restrict__ src, u64* __restrict__ dstB,
                       int L, u32 ns, const u64* __restrict__ cst, u64* side) {
  if constexpr (K > 0) {
    if (blockIdx.x < ns) {
      const int layer = blockIdx.x * blockDim.x + threadIdx.x;
      if (layer < L) lift_side<K, KB, PM>(A, src, layer, cst, side);
      return;
    }
  }
  constexpr int MQ = K ? K : PEPSI_MAXQ, MB = KB ? KB : PEPSI_MAXB;
  const int N = A.N, k = K ? K : A.k, kb = KB ? KB : A.kb;
  const size_t idx = (size_t)(blockIdx.x - ns) * blockDim.x + threadIdx.x;  // over L*2*N
  if (idx >= (size_t)L * 2 * N) return;
  const int n = (int)(idx % N);
  const size_t lc = idx / N;  // layer*2 + comp
  u64 x[MQ], v[MQ];
#pragma unroll
  for (int i = 0; i < MQ; ++i)
    if (K || i < k) x[i] = src[(lc * k + i) * N + n];
  garner_q<K, PM>(A, x, v);
  const bool neg = digits_greater<MQ>(v, A.rc.qhalf_dig, k);
#pragma unroll
  for (int j = 0; j < MB; ++j)
    if (KB || j < kb) dstB[(lc * kb + j) * N + n] = q_digits_mod_b<K, PM>(A, v, neg, j);
}

template <bool PM>
__global__ void k_lift_side(const __grid_constant__ RnsArgs A, const u64* __restrict__ src, int L,
                            const u64* __restrict__ cst, u64* side) {
  const int layer = blockIdx.x * blockDim.x + threadIdx.x;
  if (layer < L) lift_side<0, 0, PM>(A, src, layer, cst, side);
}

// ------------------------------------------------------ scale and round
// Bound by the heavy multiply-add pipe (k_lift too): a thread per coefficient holds
// its digits in registers, and with folding products the Garner and Horner steps
// stay unreduced.  A paper-shaped evaluation's scale-and-round 1.07 -> 0.72 ms, lift
// 0.61 -> 0.47 ms against Shoup and Barrett steps.
// y = round(t x / Q) exactly: z = t x + (Q-1)/2, [z]_Q from the Q residues
// by Garner, y = (z - [z]_Q) / Q computed in B, y centred in B and mapped
// back to Q by Garner over B.
template <int K, int KB, bool PM>
__global__ void k_scale_round(const __grid_constant__ RnsArgs A, const u64* __restrict__ T3, u64* __restrict__ D,
                              int L) {
  constexpr int MQ = K ? K : PEPSI_MAXQ, MB = KB ? KB : PEPSI_MAXB;
  const int N = A.N, k = K ? K : A.k, kb = KB ? KB : A.kb, np = k + kb;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // over L*3*N
  if (idx >= (size_t)L * 3 * N) return;
  const int n = (int)(idx % N);
  const size_t lc = idx / N;
  const u64* in = T3 + lc * np * N + n;
  // t x + h mod p, PM: below 2 p + h < 3 p
  auto scaled = [&](int i, u64 t, u64 ts, u64 h) {
    const DevPrime& p = A.pr[i];
    const u64 x = in[(size_t)i * N];
    if constexpr (PM)
      return PmMul(p).mul_small(x, (u32)t) + h;
    else
      return addmod(shoup(x, t, ts, p.q), h, p.q);
  };
  u64 z[MQ], v[MQ];
#pragma unroll
  for (int i = 0; i < MQ; ++i)
    if (K || i < k) z[i] = scaled(i, A.rc.t_q[i], A.rc.t_qs[i], A.rc.qhalf_q[i]);
  garner_q<K, PM>(A, z, v);
  u64 y[MB], u[MB];
#pragma unroll
  for (int j = 0; j < MB; ++j)
    if (KB || j < kb) {
      const DevPrime& pb = A.pr[k + j];
      const u64 zb = scaled(k + j, A.rc.t_b[j], A.rc.t_bs[j], A.rc.qhalf_b[j]);
      if constexpr (PM) {
        const u64 zq = horner<MQ, PM>(v, k, A.rc.qb[j], A.rc.qbs[j], pb);  // below 4 p
        y[j] = PmMul(pb).mul(zb + 4 * pb.q - zq, A.rc.qinv_b[j], A.rc.qinv_bs[j]);
      } else {
        const u64 zq = q_digits_mod_b<K, PM>(A, v, false, j);
        y[j] = shoup(submod(zb, zq, pb.q), A.rc.qinv_b[j], A.rc.qinv_bs[j], pb.q);
      }
    }
  garner_b<K, KB, PM>(A, y, u);
  const bool neg = digits_greater<MB>(u, A.rc.bhalf_dig, kb);
  u64* out = D + lc * k * N + n;
#pragma unroll
  for (int i = 0; i < MQ; ++i)
    if (K || i < k) {
      const DevPrime& pq = A.pr[i];
      const u64 r = reduce_one<PM>(horner<MB, PM>(u, kb, A.rc.bq[i], A.rc.bqs[i], pq), pq);
      out[(size_t)i * N] = neg ? submod(r, A.rc.bmodq[i], pq.q) : r;
    }
}

}  // namespace

// instantiate F<K, KB, PM> for the prime counts in use, else the run-time generic version
// (labelled N = 16384, 8 + 10 primes, h = 8 and 100 layers: 14.35 ms an evaluation, 15.17 generic)
#define PEPSI_RNS_COUNTS(V, LAUNCH, PM)               \
  switch ((V).k * 16 + (V).kb) {                      \
    case 3 * 16 + 3: LAUNCH(3, 3, PM); break;         \
    case 3 * 16 + 4: LAUNCH(3, 4, PM); break;         \
    case 4 * 16 + 4: LAUNCH(4, 4, PM); break;         \
    case 4 * 16 + 5: LAUNCH(4, 5, PM); break;         \
    case 4 * 16 + 6: LAUNCH(4, 6, PM); break;         \
    case 8 * 16 + 8: LAUNCH(8, 8, PM); break;         \
    case 8 * 16 + 9: LAUNCH(8, 9, PM); break;         \
    case 8 * 16 + 10: LAUNCH(8, 10, PM); break;       \
    default: LAUNCH(0, 0, PM); break;                 \
  }
#define PEPSI_RNS_DISPATCH(V, LAUNCH)       \
  if ((V).host_args->rc.pm) {               \
    PEPSI_RNS_COUNTS(V, LAUNCH, true)       \
  } else {                                  \
    PEPSI_RNS_COUNTS(V, LAUNCH, false)      \
  }

void launch_lift(const DevView& V, const u64* src, u64* dstB, int L, const u64* cst, u64* side, cudaStream_t st) {
  const size_t total = (size_t)L * 2 * V.N;
  if (!total) return;
#define LIFT(KQ, KBB, PM)                                                                               \
  {                                                                                                     \
    const unsigned ns = cst && KQ ? grid_for(L, 128) : 0;                                               \
    k_lift<KQ, KBB, PM><<<ns + grid_for(total, 128), 128, 0, st>>>(*V.host_args, src, dstB, L, ns, cst, side); \
    if (cst && !KQ) k_lift_side<PM><<<grid_for(L, 32), 32, 0, st>>>(*V.host_args, src, L, cst, side);    \
  }
  PEPSI_RNS_DISPATCH(V, LIFT)
#undef LIFT
}

void launch_scale_round(const DevView& V, const u64* T3, u64* D, int L, cudaStream_t st) {
  const size_t total = (size_t)L * 3 * V.N;
  if (!total) return;
#define SCALE(KQ, KBB, PM) k_scale_round<KQ, KBB, PM><<<grid_for(total, 128), 128, 0, st>>>(*V.host_args, T3, D, L)
  PEPSI_RNS_DISPATCH(V, SCALE)
#undef SCALE
}

