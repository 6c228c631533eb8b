// Kernels of PEPSI's server evaluation (Algorithms 1, 2, 5) and the client
// steps around it (Algorithms 3, 7), for sm_103a: the multiply-accumulates of
// tables in 64-bit words, pointwise kernels and the pipe probes.  Integer work only.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <cstring>

#include "kernels.h"
#include "mbar.cuh"
#include "xform.cuh"

// SMs of the current device (cached per device).
int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev]) cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev);
  return cached[dev];
}

namespace {

// ------------------------------------------------------- fused MAC (K4)
// h'[l] = sum_j C[j] * P[l][j] pointwise in the NTT domain, for both
// ciphertext components.  A block owns TN consecutive (prime, point) words
// and LB layers.  One producer thread streams P and C tiles of JS codeword
// bits through NST shared-memory stages, each stage two tiled TMA copies
// (cp.async.bulk.tensor.3d: a TN x JS x LB box of P and a TN x 2 x JS box of
// C, completion counted on a "full" mbarrier); consumer warps release a
// stage through an "empty" mbarrier.  Boxes that cross the end of a
// dimension are zero-filled by the copy engine, and zeros add nothing.
// Each consumer thread owns one point and LPT layers.  Operands are in the
// split format (x = hi 2^s + lo, both halves below 2^32): a 64-bit product
// is three 32x32->64 multiply-adds in Karatsuba form into three 64-bit
// partial sums, folded into the reduced accumulator before they can
// overflow.  Every mbarrier
// wait is bounded (about one second); on expiry the block waits, again
// bounded, for its own copies in flight, sets *err and returns.
// It serves the plaintext chunks regenerated at evaluation, which come as
// 64-bit words with the points innermost; resident tables are stored in byte
// planes for k_mac_planes.
// Five 44 KB stages (220 KB of the 227 KB a block may hold): at the paper
// shape a fifth stage took the launch from 12.13 to 11.94 ms, while stages
// of 2, 3, 5 or 6 bits, or 16 layers a block, were no faster.
namespace mac {
constexpr int TN = 128, LB = 8, LPT = 2, JS = 4, NST = 5;
constexpr int LG = LB / LPT;                    // layer slices per block
constexpr int CONSUMER_WARPS = (TN / 32) * LG;  // 16
constexpr int THREADS = (CONSUMER_WARPS + 1) * 32;
constexpr int P_WORDS = LB * JS * TN, C_WORDS = 2 * JS * TN;
// A stage holds the plaintext tile, then the request tile and the request's
// half sums (4 bytes per word, read instead of added by every layer slice).
constexpr int PB = P_WORDS * 8, SB = PB + C_WORDS * 12;
constexpr size_t SMEM = (size_t)NST * SB + 2 * NST * 8 + 16 + 128;
}  // namespace mac

__device__ __forceinline__ void tma_load_3d(u32 dst, const CUtensorMap* tm, int c0, int c1, int c2, u32 bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          dst),
      "l"(reinterpret_cast<u64>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
// acc += a * b for 32-bit a, b into a 64-bit sum (one wide multiply-add).
// Measured on this GPU with operands that change every step: 7.0 T such
// accumulations per second (the product alone, mul.wide.u32, 18 T/s).  A
// carry-chained pair of 32-bit multiply-adds (9.5 T/s in isolation) and a
// product plus separate 64-bit adds gave no faster multiply-accumulate.
__device__ __forceinline__ void mad_wide(u64& acc, u32 a, u32 b) {
  asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// The first 128-byte boundary of the dynamic shared memory, as an offset
// from the array itself (the compiler then keeps the shared address space).
__device__ __forceinline__ unsigned char* stage_base(u64* raw) {
  const u32 a = (u32)__cvta_generic_to_shared(raw);
  return reinterpret_cast<unsigned char*>(raw) + ((128u - (a & 127u)) & 127u);
}
// Karatsuba form of a split product c x = (ch 2^s + cl)(xh 2^s + xl): three
// wide multiply-adds, S0 += cl xl, S2 += ch xh, SM += (cl + ch)(xl + xh),
// instead of four.  The middle sum S1 = sum cl xh + ch xl is SM - S0 - S2
// at the fold, exact mod 2^64: SM may wrap, S0, S1 and S2 stay below 2^64.
// (Taking S2 and SM as a product plus a separate 64-bit add, which moves
// work from the multiply-add pipe to the ALU and runs twice as fast in
// isolation, left both multiply-accumulate kernels within 3% of this form.)
__device__ __forceinline__ void kmac(u64& S0, u64& SM, u64& S2, u32 cl, u32 ch, u32 cs, u32 xl, u32 xh, u32 xs) {
  mad_wide(S0, cl, xl);
  mad_wide(S2, ch, xh);
  mad_wide(SM, cs, xs);
}
// S0 + (SM - S0 - S2) 2^s + S2 2^2s as a 128-bit value (hi, lo)
__device__ __forceinline__ void compose(u64 S0, u64 SM, u64 S2, u64 s, u64& hi, u64& lo) {
  const u64 S1 = SM - S0 - S2;
  lo = S0;
  hi = 0;
  const u64 a = S1 << s;
  hi += S1 >> (64 - s);
  lo += a;
  hi += lo < a;
  const u64 b = S2 << (2 * s);
  hi += S2 >> (64 - 2 * s);
  lo += b;
  hi += lo < b;
}
// The sums reduced mod q back into S0 and SM (S2 = 0): both restart at the
// residue r, so SM - S0 stays the middle term; the fold interval leaves
// room for r below 2^64.
__device__ __forceinline__ void fold_inplace(u64& S0, u64& SM, u64& S2, u64 s, const DevPrime& pr) {
  u64 hi, lo;
  compose(S0, SM, S2, s, hi, lo);
  S0 = SM = reduce128(hi, lo, pr);
  S2 = 0;
}
__device__ __forceinline__ void fold_into(u64& acc, u64& S0, u64& SM, u64& S2, u64 s, const DevPrime& pr) {
  u64 hi, lo;
  compose(S0, SM, S2, s, hi, lo);
  acc = addmod(acc, reduce128(hi, lo, pr), pr.q);
  S0 = SM = S2 = 0;
}

__global__ void __launch_bounds__(mac::THREADS, 1)
    k_mac(DevView V, const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmC,
          const __grid_constant__ CUtensorMap tmS, u64* __restrict__ H, int ell, int L, int fold_stages, int* err) {
  using namespace mac;
  extern __shared__ __align__(128) u64 sm_raw[];
  // 128-byte aligned stage buffers for the tensor copies, derived from the
  // shared array by pointer arithmetic so that its loads stay shared-memory
  // loads
  unsigned char* sm = stage_base(sm_raw);
  const size_t kN = (size_t)V.k * V.N;
  const int l0 = blockIdx.x * LB;
  const int nl = min(LB, L - l0);
  const size_t idx0 = (size_t)blockIdx.y * TN;
  const int cnt = (int)min((size_t)TN, kN - idx0);
  const int nst = (ell + JS - 1) / JS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 sbase = (u32)__cvta_generic_to_shared(sm);
  const u32 full0 = sbase + (u32)(NST * SB), empty0 = full0 + NST * 8;
  int* abort_flag = reinterpret_cast<int*>(sm + NST * SB + 2 * NST * 8);
  if (threadIdx.x == 0) {
    for (int b = 0; b < NST; ++b) {
      mbar_init(full0 + 8 * b, 1);
      mbar_init(empty0 + 8 * b, CONSUMER_WARPS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  int issued = 0;  // producer: stages issued
  if (warp == CONSUMER_WARPS) {
    // ---------------- producer: one thread issues the tensor copies of each stage
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&tmP)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&tmC)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&tmS)) : "memory");
      for (int st = 0; st < nst; ++st) {
        const int buf = st % NST;
        if (st >= NST && !mbar_wait_bounded(empty0 + 8 * buf, (u32)(((st / NST) - 1) & 1))) {
          ok = false;
          break;
        }
        const u32 bar = full0 + 8 * buf;
        const u32 sb = sbase + (u32)(buf * SB);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, (u32)SB);
        tma_load_3d(sb, &tmP, (int)idx0, st * JS, l0, bar);
        tma_load_3d(sb + (u32)PB, &tmC, (int)idx0, 0, st * JS, bar);
        tma_load_3d(sb + (u32)(PB + C_WORDS * 8), &tmS, (int)idx0, 0, st * JS, bar);
        issued = st + 1;
      }
    }
  } else {
    // ---------------- consumer warps
    const int tp = (warp % (TN / 32)) * 32 + lane;  // point within the tile
    const int g = warp / (TN / 32);                 // layer slice
    const bool active = tp < cnt;
    const size_t idx = idx0 + (active ? tp : 0);
    const DevPrime pr = V.pr[idx / V.N];
    const u64 sp = pr.split;
    u64 S0[LPT][2], SM[LPT][2], S2[LPT][2], acc[LPT][2];
#pragma unroll
    for (int l = 0; l < LPT; ++l)
#pragma unroll
      for (int c = 0; c < 2; ++c) S0[l][c] = SM[l][c] = S2[l][c] = acc[l][c] = 0;
    int since = 0;
    for (int st = 0; st < nst; ++st) {
      const int buf = st % NST;
      if (!mbar_wait_bounded(full0 + 8 * buf, (u32)((st / NST) & 1))) {
        ok = false;
        break;
      }
      const unsigned char* stg = sm + (size_t)buf * SB;
      const u64* ps = reinterpret_cast<const u64*>(stg) + g * LPT * JS * TN + tp;  // (slice, bit 0, point)
      const u64* cs = reinterpret_cast<const u64*>(stg + PB) + tp;
      const u32* ss = reinterpret_cast<const u32*>(stg + PB + C_WORDS * 8) + tp;
#pragma unroll
      for (int jj = 0; jj < JS; ++jj) {
        const u64 c0 = cs[(jj * 2) * TN], c1 = cs[(jj * 2 + 1) * TN];
        const u32 c0l = (u32)c0, c0h = (u32)(c0 >> 32), c1l = (u32)c1, c1h = (u32)(c1 >> 32);
        const u32 c0s = ss[(jj * 2) * TN], c1s = ss[(jj * 2 + 1) * TN];
#pragma unroll
        for (int l = 0; l < LPT; ++l) {
          const u64 x = ps[(l * JS + jj) * TN];
          const u32 xl = (u32)x, xh = (u32)(x >> 32), xs = xl + xh;
          kmac(S0[l][0], SM[l][0], S2[l][0], c0l, c0h, c0s, xl, xh, xs);
          kmac(S0[l][1], SM[l][1], S2[l][1], c1l, c1h, c1s, xl, xh, xs);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8 * buf);
      if (++since == fold_stages) {
#pragma unroll
        for (int l = 0; l < LPT; ++l)
#pragma unroll
          for (int c = 0; c < 2; ++c) fold_into(acc[l][c], S0[l][c], SM[l][c], S2[l][c], sp, pr);
        since = 0;
      }
    }
    if (ok && active) {
#pragma unroll
      for (int l = 0; l < LPT; ++l)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          fold_into(acc[l][c], S0[l][c], SM[l][c], S2[l][c], sp, pr);
          const int layer = g * LPT + l;
          if (layer < nl) H[((size_t)(l0 + layer) * 2 + c) * kN + idx] = acc[l][c];
        }
    }
  }
  if (!ok) atomicExch(abort_flag, 1);
  __syncthreads();
  if (*abort_flag && warp == CONSUMER_WARPS && lane == 0) {
    // copies of the last NST issued stages may still be landing: wait for them
    for (int st = max(0, issued - NST); st < issued; ++st)
      mbar_wait_bounded(full0 + 8 * (st % NST), (u32)((st / NST) & 1));
    atomicExch(err, 1);
  }
}

// Multi-request variant: QB <= 4 requests against the same plaintexts.
// Each plaintext tile is read from HBM once and feeds 2*QB products per
// word, so the batch's plaintext stream costs what one request's does and
// the kernel is bound by the wide multiply-adds instead (6 per plaintext
// word and request).  A block owns TN = 32*WPS consecutive (prime, point)
// words and LB = 16/WPS layers.  Each of the 8 consumer warps covers 32
// points of one layer slice; each consumer thread one point, LPT = 2 layers
// and all QB requests: a plaintext word loaded from shared memory serves
// 2*QB products and a request word (with its half sum) LPT products, so a
// 4-request batch reads 10 shared-memory words and 8 half sums per 48
// multiply-adds (the SM's shared-memory bandwidth is a quarter of its wide
// multiply-add rate in 8-byte words).
// Its 48 64-bit partial sums per thread are why there are 8 consumer warps:
// with the producer, 9 warps put at most 3 on an SM sub-partition, whose
// 16K registers then allow 168 per thread (13 warps would cap them at
// 128 and spill).  Each request's tile is two 3-D TMA boxes (points x
// components x bits: its split words and their half sums, plain loads of
// this GPU's memory).  Same
// pipeline, split operands, Karatsuba sums, folding and bounded waits as
// k_mac.  Each request has its own tensor map and output, so the requests
// may live anywhere; the tile width WPS is a schedule choice (wider rows per copy
// against fewer re-reads of the request tiles, which every layer group
// reads again from L2).
namespace macq {
constexpr int LPT = 2, JS = 4, NST = 4, QMAX = 4, GROUP_WARPS = 8;
static_assert(QMAX == PEPSI_MAC_MAX_REQUESTS, "one request bound");
// RG request groups of GROUP_WARPS consumer warps each, plus the producer warp
__host__ __device__ constexpr int threads(int RG) { return (GROUP_WARPS * RG + 1) * 32; }
template <int WPS>
struct Tile {
  static constexpr int TN = 32 * WPS;                // points per block
  static constexpr int LG = GROUP_WARPS / WPS;       // layer slices
  static constexpr int LB = LG * LPT;                // layers per block
  static constexpr int P_WORDS = LB * JS * TN;
  static_assert(LG * WPS == GROUP_WARPS, "whole layer slices");
};
// request q's tile of split words, then its tile of half sums
template <int WPS>
__host__ __device__ constexpr int req_bytes() {
  return 2 * JS * Tile<WPS>::TN * 12;
}
template <int QB, int WPS>
__host__ __device__ constexpr int stage_bytes() {
  return Tile<WPS>::P_WORDS * 8 + QB * req_bytes<WPS>();
}
template <int QB, int WPS>
__host__ __device__ constexpr size_t smem() {
  return (size_t)NST * stage_bytes<QB, WPS>() + 2 * NST * 8 + 16 + 128;
}
}  // namespace macq

template <int QB, int RG, int WPS>
__global__ void __launch_bounds__(macq::threads(RG), 1)
    k_mac_multi(DevView V, const __grid_constant__ CUtensorMap tmP, const __grid_constant__ MacRequests rq, int ell,
                int L, int fold_stages, int* err) {
  using namespace macq;
  using TL = Tile<WPS>;
  constexpr int CONSUMER_WARPS = GROUP_WARPS * RG, QT = QB / RG;  // QT requests per consumer thread
  static_assert(QT * RG == QB, "whole request groups");
  constexpr int TN = TL::TN, LB = TL::LB, PW = TL::P_WORDS;
  constexpr int SB = stage_bytes<QB, WPS>(), PB = PW * 8;
  extern __shared__ __align__(128) u64 sm_raw[];
  unsigned char* sm = stage_base(sm_raw);
  const size_t kN = (size_t)V.k * V.N;
  const int l0 = blockIdx.x * LB;
  const int nl = min(LB, L - l0);
  const size_t idx0 = (size_t)blockIdx.y * TN;
  const int cnt = (int)min((size_t)TN, kN - idx0);
  const int nst = (ell + JS - 1) / JS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 sbase = (u32)__cvta_generic_to_shared(sm);
  const u32 full0 = sbase + (u32)(NST * SB), empty0 = full0 + NST * 8;
  int* abort_flag = reinterpret_cast<int*>(sm + NST * SB + 2 * NST * 8);
  if (threadIdx.x == 0) {
    for (int b = 0; b < NST; ++b) {
      mbar_init(full0 + 8 * b, 1);
      mbar_init(empty0 + 8 * b, CONSUMER_WARPS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  int issued = 0;
  if (warp == CONSUMER_WARPS) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&tmP)) : "memory");
#pragma unroll
      for (int q = 0; q < QB; ++q) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&rq.c[q])) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<u64>(&rq.s[q])) : "memory");
      }
      for (int st = 0; st < nst; ++st) {
        const int buf = st % NST;
        if (st >= NST && !mbar_wait_bounded(empty0 + 8 * buf, (u32)(((st / NST) - 1) & 1))) {
          ok = false;
          break;
        }
        const u32 bar = full0 + 8 * buf;
        const u32 sb = sbase + (u32)(buf * SB);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, (u32)SB);
        tma_load_3d(sb, &tmP, (int)idx0, st * JS, l0, bar);
#pragma unroll
        for (int q = 0; q < QB; ++q) {
          const u32 rb = sb + (u32)(PB + q * req_bytes<WPS>());
          tma_load_3d(rb, &rq.c[q], (int)idx0, 0, st * JS, bar);
          tma_load_3d(rb + (u32)(2 * JS * TN * 8), &rq.s[q], (int)idx0, 0, st * JS, bar);
        }
        issued = st + 1;
      }
    }
  } else {
    const int rg = warp / GROUP_WARPS, gw = warp % GROUP_WARPS;  // request group, warp within it
    const int tp = (gw % WPS) * 32 + lane;  // point within the tile
    const int g = gw / WPS;                 // layer slice
    const bool active = tp < cnt;
    const size_t idx = idx0 + (active ? tp : 0);
    const DevPrime pr = V.pr[idx / V.N];
    const u64 sp = pr.split;
    u64 S0[LPT][QT][2], SM[LPT][QT][2], S2[LPT][QT][2];
#pragma unroll
    for (int l = 0; l < LPT; ++l)
#pragma unroll
      for (int q = 0; q < QT; ++q)
#pragma unroll
        for (int c = 0; c < 2; ++c) S0[l][q][c] = SM[l][q][c] = S2[l][q][c] = 0;
    int since = 0;
    for (int st = 0; st < nst; ++st) {
      const int buf = st % NST;
      if (!mbar_wait_bounded(full0 + 8 * buf, (u32)((st / NST) & 1))) {
        ok = false;
        break;
      }
      const unsigned char* stg = sm + (size_t)buf * SB;
      const u64* ps = reinterpret_cast<const u64*>(stg) + g * LPT * JS * TN + tp;  // (slice, bit 0, point)
      const unsigned char* rqt = stg + PB + rg * QT * req_bytes<WPS>();  // this group's request tiles
#pragma unroll
      for (int jj = 0; jj < JS; ++jj) {
        u32 xl[LPT], xh[LPT], xs[LPT];
#pragma unroll
        for (int l = 0; l < LPT; ++l) {
          const u64 x = ps[(l * JS + jj) * TN];
          xl[l] = (u32)x;
          xh[l] = (u32)(x >> 32);
          xs[l] = xl[l] + xh[l];
        }
#pragma unroll
        for (int q = 0; q < QT; ++q)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const unsigned char* t = rqt + q * req_bytes<WPS>();
            const u64 w = reinterpret_cast<const u64*>(t)[(jj * 2 + c) * TN + tp];
            const u32 cl = (u32)w, ch = (u32)(w >> 32);
            const u32 csum = reinterpret_cast<const u32*>(t + 2 * JS * TN * 8)[(jj * 2 + c) * TN + tp];
#pragma unroll
            for (int l = 0; l < LPT; ++l)
              kmac(S0[l][q][c], SM[l][q][c], S2[l][q][c], cl, ch, csum, xl[l], xh[l], xs[l]);
          }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8 * buf);
      if (++since == fold_stages) {
#pragma unroll
        for (int l = 0; l < LPT; ++l)
#pragma unroll
          for (int q = 0; q < QT; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) fold_inplace(S0[l][q][c], SM[l][q][c], S2[l][q][c], sp, pr);
        since = 0;
      }
    }
    if (ok && active) {
#pragma unroll
      for (int l = 0; l < LPT; ++l)
#pragma unroll
        for (int q = 0; q < QT; ++q)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            fold_inplace(S0[l][q][c], SM[l][q][c], S2[l][q][c], sp, pr);
            const int layer = g * LPT + l;
            if (layer < nl) rq.h[rg * QT + q][((size_t)(l0 + layer) * 2 + c) * kN + idx] = S0[l][q][c];
          }
    }
  }
  if (!ok) atomicExch(abort_flag, 1);
  __syncthreads();
  if (*abort_flag && warp == CONSUMER_WARPS && lane == 0) {
    for (int st = max(0, issued - NST); st < issued; ++st)
      mbar_wait_bounded(full0 + 8 * (st % NST), (u32)((st / NST) & 1));
    atomicExch(err, 1);
  }
}

// In-place conversion of [rows][N] words between the reduced and the split
// operand format; row r uses prime r % k.
__global__ void k_split(DevView V, u64* x, size_t total, int to) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const u64 s = V.pr[(i / V.N) % V.k].split;
  x[i] = to ? to_split(x[i], s) : from_split(x[i], s);
}

// ------------------------------------------------------------ pointwise
__global__ void k_axpy(DevView V, const u64* __restrict__ a, const u64* __restrict__ zres, const u64* __restrict__ b,
                       u64* out, size_t total) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int p = (int)((idx / V.N) % V.k);
  const DevPrime pr = V.pr[p];
  out[idx] = addmod(a[idx], mulmod(zres[p], b[idx], pr), pr.q);
}

__global__ void k_accum(DevView V, const u64* __restrict__ D, int L, u64* acc, int init) {
  const size_t per = (size_t)3 * V.k * V.N;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= per) return;
  const u64 q = V.pr[(idx / V.N) % V.k].q;
  u64 s = init ? 0 : acc[idx];
  for (int l = 0; l < L; ++l) s = addmod(s, D[(size_t)l * per + idx], q);
  acc[idx] = s;
}

}  // namespace

// ------------------------------------------------------------ launchers
namespace {
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}
// 3-D tensor of elements of esz bytes: dims (d0, d1, d2), row strides s1, s2 in elements, box (b0, b1, b2)
bool encode3d_t(CUtensorMap* tm, CUtensorMapDataType dt, int esz, const void* base, u64 d0, u64 d1, u64 d2, u64 s1,
                u64 s2, u32 b0, u32 b1, u32 b2) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {s1 * esz, s2 * esz};
  const cuuint32_t box[3] = {b0, b1, b2};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(tm, dt, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool encode3d(CUtensorMap* tm, const u64* base, u64 d0, u64 d1, u64 d2, u64 s1, u64 s2, u32 b0, u32 b1, u32 b2) {
  return encode3d_t(tm, CU_TENSOR_MAP_DATA_TYPE_UINT64, 8, base, d0, d1, d2, s1, s2, b0, b1, b2);
}
}  // namespace

namespace {
template <int QB, int RG, int WPS>
void mac_multi_go(const DevView& V, const CUtensorMap& tmP, const MacRequests& rq, int ell, int L, int fold_stages,
                  int* err, cudaStream_t st) {
  using TL = macq::Tile<WPS>;
  const u64 kN = (u64)V.k * V.N;
  dim3 grid((L + TL::LB - 1) / TL::LB, (unsigned)((kN + TL::TN - 1) / TL::TN));
  k_mac_multi<QB, RG, WPS><<<grid, macq::threads(RG), macq::smem<QB, WPS>(), st>>>(V, tmP, rq, ell, L, fold_stages,
                                                                                   err);
}
// groups: 1 = every consumer thread serves all requests; 2 = two groups of
// warps serve half of them each (2 or 4 requests)
template <int WPS>
void mac_multi_q(int nq, int groups, const DevView& V, const CUtensorMap& tmP, const MacRequests& rq, int ell, int L,
                 int fold_stages, int* err, cudaStream_t st) {
  switch (nq * 4 + (groups == 2 && nq != 3 ? 2 : 1)) {
    case 2 * 4 + 1: mac_multi_go<2, 1, WPS>(V, tmP, rq, ell, L, fold_stages, err, st); break;
    case 2 * 4 + 2: mac_multi_go<2, 2, WPS>(V, tmP, rq, ell, L, fold_stages, err, st); break;
    case 3 * 4 + 1: mac_multi_go<3, 1, WPS>(V, tmP, rq, ell, L, fold_stages, err, st); break;
    case 4 * 4 + 1: mac_multi_go<4, 1, WPS>(V, tmP, rq, ell, L, fold_stages, err, st); break;
    default: mac_multi_go<4, 2, WPS>(V, tmP, rq, ell, L, fold_stages, err, st); break;
  }
}
}  // namespace

cudaError_t launch_mac_requests(const DevView& V, int nq, const u64* const* C, const u64* P, u64* const* H, int ell,
                                int L, int fold, int* err, cudaStream_t st, int tile_points, int groups) {
  if (L <= 0 || nq <= 0) return cudaSuccess;
  if (nq > macq::QMAX || (tile_points != 32 && tile_points != 64)) return cudaErrorInvalidValue;
  if (nq == 1) return launch_mac(V, C[0], P, H[0], ell, L, fold, err, st);  // one request: the single-request kernel
  const u64 kN = (u64)V.k * V.N;
  const int wps = tile_points / 32;
  const u32 tn = (u32)tile_points, lb = (u32)(macq::GROUP_WARPS / wps * macq::LPT);
  CUtensorMap tmP;
  MacRequests rq;
  memset(&rq, 0, sizeof(rq));
  if (!encode3d(&tmP, P, kN, ell, L, kN, (u64)ell * kN, tn, macq::JS, lb)) return cudaErrorInvalidValue;
  for (int q = 0; q < nq; ++q) {
    if (!encode3d(&rq.c[q], C[q], kN, 2, ell, kN, 2 * kN, tn, 2, macq::JS) ||
        !encode3d_t(&rq.s[q], CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, request_sums(C[q], ell, kN), kN, 2, ell, kN, 2 * kN, tn,
                    2, macq::JS))
      return cudaErrorInvalidValue;
    rq.h[q] = H[q];
  }
  const int fold_stages = fold / macq::JS > 0 ? fold / macq::JS : 1;
  if (wps == 1)
    mac_multi_q<1>(nq, groups, V, tmP, rq, ell, L, fold_stages, err, st);
  else
    mac_multi_q<2>(nq, groups, V, tmP, rq, ell, L, fold_stages, err, st);
  return cudaSuccess;
}

cudaError_t launch_mac(const DevView& V, const u64* C, const u64* P, u64* H, int ell, int L, int fold, int* err,
                       cudaStream_t st) {
  if (L <= 0) return cudaSuccess;
  const u64 kN = (u64)V.k * V.N;
  CUtensorMap tmP, tmC, tmS;
  if (!encode3d(&tmP, P, kN, ell, L, kN, (u64)ell * kN, mac::TN, mac::JS, mac::LB) ||
      !encode3d(&tmC, C, kN, 2, ell, kN, 2 * kN, mac::TN, 2, mac::JS) ||
      !encode3d_t(&tmS, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, request_sums(C, ell, kN), kN, 2, ell, kN, 2 * kN, mac::TN, 2,
                  mac::JS))
    return cudaErrorInvalidValue;
  const int fold_stages = fold / mac::JS > 0 ? fold / mac::JS : 1;
  dim3 grid((L + mac::LB - 1) / mac::LB, (unsigned)((kN + mac::TN - 1) / mac::TN));
  k_mac<<<grid, mac::THREADS, mac::SMEM, st>>>(V, tmP, tmC, tmS, H, ell, L, fold_stages, err);
  return cudaSuccess;
}

void launch_split(const DevView& V, u64* x, size_t groups, bool to, cudaStream_t st) {
  const size_t total = groups * V.k * V.N;
  if (!total) return;
  k_split<<<grid_for(total, 256), 256, 0, st>>>(V, x, total, to ? 1 : 0);
}

// Value-weighted layer sum with per-layer rounding: acc[c][p][n] (+)=
// sum_{l<L} D_l[c][p][n] * VP_l[p][n] mod q_p, D in NTT form over Q.  One
// product below 2^122 per layer; the 128-bit sums are reduced every 32.
__global__ void k_accum_val(DevView V, const u64* __restrict__ D, const u64* __restrict__ VP, int L, u64* acc,
                            int init) {
  const int N = V.N, k = V.k, np = V.k + V.kb;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // over 3*k*N
  if (idx >= (size_t)3 * k * N) return;
  const int n = (int)(idx % N);
  const int p = (int)((idx / N) % k);
  const int c = (int)(idx / ((size_t)k * N));
  const DevPrime pr = V.pr[p];
  u64 lo = 0, hi = 0;
  for (int l = 0; l < L; ++l) {
    mac128(lo, hi, D[(((size_t)l * 3 + c) * k + p) * N + n], VP[((size_t)l * np + p) * N + n]);
    if ((l & 31) == 31) {
      lo = reduce128(hi, lo, pr);
      hi = 0;
    }
  }
  const u64 r = reduce128(hi, lo, pr);
  acc[idx] = init ? r : addmod(r, acc[idx], pr.q);
}

void launch_accum_val(const DevView& V, const u64* D, const u64* VP, int L, u64* acc, bool init, cudaStream_t st) {
  const size_t total = (size_t)3 * V.k * V.N;
  k_accum_val<<<grid_for(total, 256), 256, 0, st>>>(V, D, VP, L, acc, init ? 1 : 0);
}

void launch_axpy(const DevView& V, const u64* a, const u64* zres, const u64* b, u64* out, size_t groups,
                 cudaStream_t st) {
  const size_t total = groups * V.k * V.N;
  if (!total) return;
  k_axpy<<<grid_for(total, 256), 256, 0, st>>>(V, a, zres, b, out, total);
}

void launch_accum(const DevView& V, const u64* D, int L, u64* acc, bool init, cudaStream_t st) {
  const size_t total = (size_t)3 * V.k * V.N;
  k_accum<<<grid_for(total, 256), 256, 0, st>>>(V, D, L, acc, init ? 1 : 0);
}

// Test of the multiply-accumulate's bounded wait (mbar_wait_bounded): one thread waits on an mbarrier that
// needs one arrival.  With arrive != 0 it arrives first and the wait
// completes; with arrive == 0 nothing completes the phase, the wait gives
// up after about one second and the kernel sets *err and returns, as the
// multiply-accumulate does when its copies never land.
__global__ void k_wait_probe(int arrive, int* err) {
  __shared__ __align__(8) u64 bar;
  const u32 addr = (u32)__cvta_generic_to_shared(&bar);
  if (threadIdx.x == 0) {
    mbar_init(addr, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (arrive) mbar_arrive(addr);
    if (!mbar_wait_bounded(addr, 0)) atomicExch(err, 1);
  }
}

void launch_wait_probe(int arrive, int* err, cudaStream_t st) { k_wait_probe<<<1, 32, 0, st>>>(arrive, err); }

cudaError_t kernels_init(int N) {
  cudaError_t e = client_init(N);
  if (e == cudaSuccess) e = transforms_init();
  if (e == cudaSuccess) e = tensor_init();
  if (e == cudaSuccess) e = relin_init();
  if (e == cudaSuccess) e = mac_planes_init();
  auto set = [&](const void* f) {
    if (e == cudaSuccess) e = allow_smem(f);
  };
  set((const void*)k_mac);
#define PEPSI_SET_MACQ(QB, RG)               \
  set((const void*)k_mac_multi<QB, RG, 1>);  \
  set((const void*)k_mac_multi<QB, RG, 2>);
  PEPSI_SET_MACQ(2, 1)
  PEPSI_SET_MACQ(2, 2)
  PEPSI_SET_MACQ(3, 1)
  PEPSI_SET_MACQ(4, 1)
  PEPSI_SET_MACQ(4, 2)
#undef PEPSI_SET_MACQ
  return e;
}

// ------------------------------------------------------ integer-pipe peak
// Throughput probe of the multiply forms the kernels above are built from:
// FORM 1, 32x32->64 wide multiply-add into a 64-bit sum (mad.wide.u32, the
// multiply-accumulate's operation); FORM 2, the wide product alone
// (mul.wide.u32); FORM 0, 32-bit multiply-add (mad.lo.u32).  Each thread runs
// 16 chains; the multiplier of chain i is the low word of chain i+5, so it
// changes every step and no product can be hoisted out of the loop.  The
// result is folded into *sink so nothing is dead code.
namespace {
template <int FORM>
__global__ void k_int_peak(int iters, u32 seed, u64* sink) {
  u64 a[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = seed + threadIdx.x * 7 + i;
  const u32 m = seed | 1u;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const u32 x = (u32)a[(i + 5) & 15];
      if (FORM == 1) {
        asm volatile("mad.wide.u32 %0, %1, %2, %0;" : "+l"(a[i]) : "r"(x), "r"(m));
      } else if (FORM == 2) {
        asm volatile("mul.wide.u32 %0, %1, %2;" : "=l"(a[i]) : "r"(x), "r"(m));
      } else {
        u32 l = (u32)a[i];
        asm volatile("mad.lo.u32 %0, %1, %2, %0;" : "+r"(l) : "r"(x), "r"(m));
        a[i] = (a[i] & 0xffffffff00000000ull) | l;
      }
    }
  }
  u64 acc = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) acc += a[i];
  if (acc == 0x123456789ull) *sink = acc;
}
}  // namespace

double measure_int_peak(int form) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  u64* sink = nullptr;
  if (cudaMalloc(&sink, sizeof(u64)) != cudaSuccess) return 0;
  const int threads = 512, blocks = sms * 4, iters = 4096;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  double best = 0;
  for (int rep = 0; rep < 3; ++rep) {
    cudaEventRecord(e0);
    if (form == 1)
      k_int_peak<1><<<blocks, threads>>>(iters, 7u + rep, sink);
    else if (form == 2)
      k_int_peak<2><<<blocks, threads>>>(iters, 7u + rep, sink);
    else
      k_int_peak<0><<<blocks, threads>>>(iters, 7u + rep, sink);
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    const double ops = (double)blocks * threads * iters * 16;
    if (ms > 0) best = std::max(best, ops / (ms * 1e-3));
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(sink);
  return best;
}
