// The multiply-accumulate of a resident server table (Algorithm 1's h' = sum_j
// x_j y_j, pointwise in the NTT domain) on the tensor cores, and the byte
// plane formats it reads.
//
// For one point (prime, NTT position) the work is a matrix product:
// layers x code bits (plaintexts) times code bits x components (request).  Its
// 64-bit modular products are built from bytes.  A byte b as the 16-bit pattern
// 0x00bb is the f16 subnormal b 2^-24, exactly, so zero-extended bytes are
// already f16 operands: no conversion, only a byte permute.  Products of two
// are exact, and the f32 accumulators start at 2^23 (in units of 2^-48) so that
// a sum of up to 128 products (128 * 255^2 < 2^23) stays in [2^23, 2^24), where
// f32 holds every integer: its bit pattern minus that of 2^23 IS the sum.
// Every 128 code bits the sums move to 32-bit integer accumulators (65535 * 255^2
// < 2^32 covers every code length the library accepts).  So plane i of the
// plaintext times byte n of the request gives D[i][n] exactly, and
// h' = sum_{i,n} 2^(8 (i + n)) D[i][n] mod q.
//
// Formats (built once per table / per request):
//  - Table, NPL = ceil(bits(q)/8) bytes per word (7 for 55-bit primes instead of
//    a 64-bit word): tiles of 16 layers; inside a tile [point][step][layer] rows
//    of 16 code bits, [t < 4][plane i][4 bytes: bits 16 step + 4 t + (0..3)].
//    A thread of the 16x8x16 matrix instruction holds operand columns 2t, 2t+1,
//    2t+8, 2t+9; which code bit a column carries is free as long as both
//    operands agree, so bytes 0, 2 of a 32-bit word are one operand register
//    and bytes 1, 3 the other: one byte permute each.
//  - Request: [point][step][byte n < 8][t < 4][component][4 bytes], the same bit order.
#include <algorithm>

#include "kernels.h"
#include "mbar.cuh"

namespace {

namespace macp {
// Consumer warps: 8 with 168 registers a thread, or 12 with 128 for the kernel
// of short codes, which keeps one set of sums and is bound by what an item costs
// beside its products.
__host__ __device__ constexpr int consumers(bool brief) { return brief ? 12 : 8; }
constexpr int PRODUCERS = 4;
__host__ __device__ constexpr int threads(bool brief) { return (consumers(brief) + PRODUCERS) * 32; }
// Steps per pipeline stage.  One request streams from HBM: stages of 4 steps
// (8 KB with 7 planes), two per team, keep 128 KB on their way to an SM, and more
// only disorders the DRAM (10.4 ms at the paper shape; three stages 11.4, stages
// of 3, 5 or 6 steps 10.9, 10.5, 10.9).  Several requests are bound by the consumer
// warps, which longer stages free of waits (four requests, 48 layers: 2.76, 2.60,
// 2.46 ms at 4, 6, 8 steps).  Codes of at most 128 bits: a stage costs its producer
// warp, which serves three teams, about as much as two steps cost a consumer, so
// stages of 4 steps as well (512 layers of 128 bits at N = 8192, 7 planes: 2.41 ms,
// 2.88 with stages of 2; N = 4096, 5 planes: 0.64, 1.05).
constexpr int KS_ONE = 4, KS_MANY = 8;
constexpr int MAX_STAGES = 16;
constexpr int DRAIN = 8;           // steps between moves to the integer sums: 128 code bits
constexpr u32 BIAS = 0x33000000u;  // 2^23 in units of 2^-48, as f32
constexpr int SMEM_BUDGET = 220 * 1024;
__host__ __device__ constexpr int row_bytes(int npl) { return 16 * npl; }
// a pipeline stage: ks steps of the table tile, then of each request
__host__ __device__ constexpr int stage_bytes(int npl, int ks, int nq) { return ks * (16 * row_bytes(npl) + 256 * nq); }
}  // namespace macp

struct PlaneArgs {
  const unsigned char* P;  // table of `rows` layers
  u32 rows;
  int l0, nl;              // layers evaluated; h' of layer l0 goes to row 0 of H
  int nks, ks0, ks1;       // steps of the code, and those of this launch
  int acc_in;              // add to the h' already in H
  int nq, nst;             // requests, pipeline stages per team
  int* err;
  const u32* C[PEPSI_MAC_MAX_REQUESTS];
  u64* H[PEPSI_MAC_MAX_REQUESTS];
};

__device__ __forceinline__ void bulk_load(u32 dst, const void* src, u32 bytes, u32 bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bulk_load(u32 dst, const void* src, u32 bytes, u32 bar, u64 policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void mma_f16(float (&d)[4], u32 a0, u32 a1, u32 a2, u32 a3, u32 b0, u32 b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// bytes 0, 2 (even) or 1, 3 (odd) of a word, zero-extended to two halves
__device__ __forceinline__ u32 even_halves(u32 w) { return __byte_perm(w, 0, 0x4240); }
__device__ __forceinline__ u32 odd_halves(u32 w) { return __byte_perm(w, 0, 0x4341); }

// The NPL plane words of one (layer, thread column): widest loads its alignment allows.
template <int NPL>
__device__ __forceinline__ void load_row(u32 (&r)[NPL], const unsigned char* p) {
  if constexpr (NPL % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NPL; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(p + 4 * i);
      r[i] = v.x;
      r[i + 1] = v.y;
      r[i + 2] = v.z;
      r[i + 3] = v.w;
    }
  } else if constexpr (NPL % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NPL; i += 2) {
      const uint2 v = *reinterpret_cast<const uint2*>(p + 4 * i);
      r[i] = v.x;
      r[i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NPL; ++i) r[i] = *reinterpret_cast<const u32*>(p + 4 * i);
  }
}

struct Wide {  // lo + 2^64 hi
  u64 lo, hi;
};
// sum over the planes of (d0 + 2^8 d1) 2^(8 i), below 2^99
template <int NPL>
__device__ __forceinline__ Wide combine(const u32 (&d0)[NPL], const u32 (&d1)[NPL]) {
  u64 part[3] = {0, 0, 0};  // weights 1, 2^24, 2^48: each below 2^58, one wide multiply-add per sum
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(part[i / 3]) : "r"(d0[i]), "r"(1 << (8 * (i % 3))));
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(part[i / 3]) : "r"(d1[i]), "r"(256 << (8 * (i % 3))));
  }
  u64 lo = part[0], hi = part[1] >> 40;
  const u64 m = part[1] << 24;
  lo += m;
  hi += lo < m;
  if constexpr (NPL > 6) {
    const u64 h = part[2] << 48;
    lo += h;
    hi += (lo < h) + (part[2] >> 16);
  }
  return {lo, hi};
}
__device__ __forceinline__ Wide shfl_xor(Wide w, int m) {
  return {__shfl_xor_sync(0xffffffffu, w.lo, m), __shfl_xor_sync(0xffffffffu, w.hi, m)};
}

__device__ __forceinline__ bool elect_one() {
  u32 p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// Walk over a team's items.  Items go tile fastest, so that the teams at work
// together share a point's request bytes in L2; a step adds the grid's stride
// without a division.
struct Walk {
  u32 x, tl;      // point, tile within the launch's
  u32 dx, dt, ntile;
  __device__ __forceinline__ Walk(u32 first, u32 stride, u32 n) : x(first / n), tl(first % n), dx(stride / n), dt(stride % n), ntile(n) {}
  __device__ __forceinline__ void next() {
    x += dx;
    tl += dt;
    if (tl >= ntile) {
      tl -= ntile;
      ++x;
    }
  }
};
// A tile: its used rows [ra, ra + nr) and stored rows R.
struct Tile {
  u32 tile;
  int ra, nr, R;
  __device__ __forceinline__ Tile(const PlaneArgs& A, u32 t) : tile(t) {
    const int first = (int)(t * 16);
    ra = max(A.l0 - first, 0);
    nr = min(A.l0 + A.nl - first, 16) - ra;
    R = min(16, (int)A.rows - first);
  }
};

// Persistent block: consumer warps in teams of nq (one warp per request), each
// team with a ring of pipeline stages and items of its own, and producer warps
// that keep up to two rings filled with bulk copies across item boundaries.
// (With the copies issued by the consumers themselves each stage cost them
// about 560 cycles of serial address work: one request took 12.1 ms instead of
// 11.1 ms at the paper shape, four requests and 48 layers 3.1 ms instead of 2.7.)
// Every wait is bounded (about one second); on expiry the warp goes on to
// where it can stop, sets *err and returns.  The producers wait, again bounded, for
// the last copies of their teams before they return.
// SHORT: at most DRAIN steps, so the integer sums are read once.
template <int NPL, int KS, bool SHORT>
__global__ void __launch_bounds__(macp::threads(SHORT), 1) k_mac_planes(DevView V, const __grid_constant__ PlaneArgs A) {
  using namespace macp;
  constexpr int RB = row_bytes(NPL), CONSUMERS = consumers(SHORT), TEAMS_PER_PRODUCER = CONSUMERS / PRODUCERS;
  extern __shared__ __align__(128) unsigned char smp[];
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int nq = A.nq, nst = A.nst, teams = CONSUMERS / nq;
  const u32 kN = (u32)V.k * V.N;
  const u32 SB = (u32)stage_bytes(NPL, KS, nq);
  const u32 base = (u32)__cvta_generic_to_shared(smp), bars = base + (u32)(teams * nst) * SB;
  auto full = [&](int team, int s) -> u32 { return bars + (u32)(team * 2 * nst + s) * 8; };
  auto empty = [&](int team, int s) -> u32 { return bars + (u32)(team * 2 * nst + nst + s) * 8; };
  if (threadIdx.x == 0) {
    for (int u = 0; u < teams; ++u)
      for (int b = 0; b < nst; ++b) {
        mbar_init(full(u, b), 1);
        mbar_init(empty(u, b), nq);
      }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const u32 tile0 = (u32)A.l0 >> 4, ntile = ((u32)(A.l0 + A.nl + 15) >> 4) - tile0;
  const u32 stride = gridDim.x * teams;
  bool ok = true;  // the same in every lane

  if (warp >= CONSUMERS) {
    // ---------------- producer: teams p and p + PRODUCERS
    const int p = warp - CONSUMERS;
    // The table is read once, a point's request by every tile: without the hint
    // the stream evicts the requests (11.1 ms against 10.4 ms at the paper shape).
    u64 stream;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream));
    const size_t tile_bytes = (size_t)16 * kN * A.nks * RB;
    const u32 first = blockIdx.x * teams + p;
    Walk w0(first, stride, ntile);
    u32 x[TEAMS_PER_PRODUCER], tl[TEAMS_PER_PRODUCER], used[TEAMS_PER_PRODUCER], step[TEAMS_PER_PRODUCER];
    int ck[TEAMS_PER_PRODUCER];
    const unsigned char* psrc[TEAMS_PER_PRODUCER];
    size_t coff[TEAMS_PER_PRODUCER];
    auto open = [&](int u) {
      const Tile T(A, tile0 + tl[u]);
      used[u] = T.nr * RB;
      step[u] = T.R * RB;
      psrc[u] = A.P + T.tile * tile_bytes + (u64)(x[u] * (u32)A.nks + (u32)A.ks0) * step[u] + T.ra * RB;
      coff[u] = (size_t)(x[u] * (u32)A.nks + (u32)A.ks0) * 64;
      ck[u] = A.ks0;
    };
#pragma unroll
    for (int u = 0; u < TEAMS_PER_PRODUCER; ++u) {
      const Walk w(first + u * PRODUCERS, stride, ntile);
      x[u] = p + u * PRODUCERS < teams ? w.x : 0xFFFFFFFFu;  // none
      tl[u] = w.tl;
      if (x[u] < kN) open(u);
    }
    int slot = 0, round = 0, last_slot[TEAMS_PER_PRODUCER] = {}, filled[TEAMS_PER_PRODUCER] = {};
    while (ok) {
      bool any = false;
#pragma unroll
      for (int u = 0; u < TEAMS_PER_PRODUCER; ++u) {
        if (x[u] >= kN || !ok) continue;
        any = true;
        const int team = p + u * PRODUCERS;
        if (round > 0) {
          ok = __all_sync(0xffffffffu, mbar_wait_bounded(empty(team, slot), (u32)(round - 1) & 1));
          if (!ok) continue;
        }
        const int kc = min(KS, A.ks1 - ck[u]);
        const u32 bar = full(team, slot), dst = base + (u32)(team * nst + slot) * SB;
        if (elect_one()) {
          mbar_expect_tx(bar, (u32)kc * (used[u] + 256u * nq));
          if (used[u] == step[u]) {
            bulk_load(dst, psrc[u], (u32)kc * step[u], bar, stream);
          } else {
            for (int s = 0; s < kc; ++s)
              bulk_load(dst + (u32)s * used[u], psrc[u] + (size_t)s * step[u], used[u], bar, stream);
          }
          for (int q = 0; q < nq; ++q)
            bulk_load(dst + (u32)(KS * (16 * RB + q * 256)), A.C[q] + coff[u], (u32)(kc * 256), bar);
        }
        filled[u] = min(filled[u] + 1, nst);
        last_slot[u] = round * nst + slot;
        ck[u] += kc;
        psrc[u] += (size_t)kc * step[u];
        coff[u] += (size_t)kc * 64;
        if (ck[u] >= A.ks1) {
          w0.x = x[u];
          w0.tl = tl[u];
          w0.next();
          x[u] = w0.x;
          tl[u] = w0.tl;
          if (x[u] < kN) open(u);
        }
      }
      if (!any) break;
      if (++slot == nst) {
        slot = 0;
        ++round;
      }
    }
    // Copies still in flight are among the last nst stages issued to each team: none
    // may land after the block has ended, also where a consumer's wait expired.
#pragma unroll
    for (int u = 0; u < TEAMS_PER_PRODUCER; ++u)
      for (int b = 0; b < filled[u]; ++b) {
        const int n = last_slot[u] - b;
        ok &= mbar_wait_bounded(full(p + u * PRODUCERS, n % nst), (u32)(n / nst) & 1);
      }
    if (!ok && lane == 0) atomicExch(A.err, 1);
    return;
  }

  // ---------------- consumer: warp `member` of a team serves request `member`
  const int team = warp / nq, member = warp - team * nq, g = lane >> 2, t = lane & 3;
  if (team >= teams) return;
  const unsigned char* const ring = smp + (size_t)team * nst * SB;
  int slot = 0;
  u32 parity = 0;
  for (Walk w(blockIdx.x * teams + team, stride, ntile); w.x < kN && ok; w.next()) {
    const Tile T(A, tile0 + w.tl);
    const int nr = T.nr;
    const int o0 = min(g, nr - 1) * RB + t * 4 * NPL, o1 = min(g + 8, nr - 1) * RB + t * 4 * NPL;
    float acc[NPL][2][4];
    u32 sum[NPL][2][4];
#pragma unroll
    for (int i = 0; i < NPL; ++i)
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[i][c][e] = __uint_as_float(BIAS);
          if (!SHORT) sum[i][c][e] = 0;
        }
    // one step: 16 layers x 16 code bits of every plane against both components
    auto step = [&](const unsigned char* stg, int s) {
      u32 r0[NPL], r1[NPL];
      load_row<NPL>(r0, stg + s * nr * RB + o0);
      load_row<NPL>(r1, stg + s * nr * RB + o1);
      const uint2 b = *reinterpret_cast<const uint2*>(stg + KS * 16 * RB + (member * KS + s) * 256 + lane * 8);
      const u32 b00 = even_halves(b.x), b01 = odd_halves(b.x), b10 = even_halves(b.y), b11 = odd_halves(b.y);
#pragma unroll
      for (int i = 0; i < NPL; ++i) {
        const u32 a0 = even_halves(r0[i]), a1 = even_halves(r1[i]), a2 = odd_halves(r0[i]), a3 = odd_halves(r1[i]);
        mma_f16(acc[i][0], a0, a1, a2, a3, b00, b01);
        mma_f16(acc[i][1], a0, a1, a2, a3, b10, b11);
      }
    };
    auto drain = [&]() {
#pragma unroll
      for (int i = 0; i < NPL; ++i)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (SHORT) {
              sum[i][c][e] = __float_as_uint(acc[i][c][e]) - BIAS;
            } else {
              sum[i][c][e] += __float_as_uint(acc[i][c][e]) - BIAS;
              acc[i][c][e] = __uint_as_float(BIAS);
            }
          }
    };
    // A warp whose wait expired goes on with stale bytes and waits no more; the
    // item is dropped below.
    auto arrive_at = [&]() {
      if (!__all_sync(0xffffffffu, mbar_try_wait(full(team, slot), parity)) && ok)
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(full(team, slot), parity));
    };
    // The stage is refilled by an asynchronous copy, which a generic read is ordered
    // before only through a proxy fence: without it the copy of the stage after next
    // overwrote rows still being read (stages of one to three steps, where a stage's
    // reads are few and its refill comes soon: a handful of wrong items in 11 million).
    // Every lane fences its own reads, which keeps the producer warp, the bound of
    // short codes, free of it; no case's time changes by more than its runs differ.
    auto leave = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();  // every lane has read the stage
      if (lane == 0) mbar_arrive(empty(team, slot));
      if (++slot == nst) {
        slot = 0;
        parity ^= 1;
      }
    };
    const int nfull = (A.ks1 - A.ks0) / KS;
    for (int i = 1; i <= nfull; ++i) {
      arrive_at();
      const unsigned char* stg = ring + (size_t)slot * SB;
#pragma unroll
      for (int s = 0; s < KS; ++s) step(stg, s);
      leave();
      if (!SHORT && i % (DRAIN / KS) == 0) drain();
    }
    if ((A.ks1 - A.ks0) % KS) {  // the last, partial stage
      arrive_at();
      const unsigned char* stg = ring + (size_t)slot * SB;
      for (int s = 0; s < (A.ks1 - A.ks0) % KS; ++s) step(stg, s);
      leave();
    }
    drain();
    if (!ok) break;
    // The thread's columns 2t, 2t+1 of four (layer, component) values v (v = 2 *
    // row half + component), weighted 2^(16 t), are summed over the quad, value
    // v by thread t = v: two exchanges in which each thread sends the values
    // the other one keeps.
    const DevPrime pr = V.pr[w.x >> V.logN];
    Wide val[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int e = (v >> 1) * 2, c = v & 1;
      u32 d0[NPL], d1[NPL];
#pragma unroll
      for (int i = 0; i < NPL; ++i) {
        d0[i] = sum[i][c][e];
        d1[i] = sum[i][c][e + 1];
      }
      val[v] = combine<NPL>(d0, d1);
    }
    Wide pairs[2];  // values v = t & 1 and 2 + (t & 1): columns of threads t & 2 and (t & 2) + 1, below 2^116
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const Wide own = t & 1 ? val[2 * u + 1] : val[2 * u];
      const Wide other = shfl_xor(t & 1 ? val[2 * u] : val[2 * u + 1], 1);
      const Wide a = t & 1 ? other : own, b = t & 1 ? own : other;  // weights 1, 2^16
      const u64 bl = b.lo << 16, lo = a.lo + bl;
      pairs[u] = {lo, a.hi + (b.hi << 16 | b.lo >> 48) + (lo < bl)};
    }
    const Wide own = t & 2 ? pairs[1] : pairs[0];
    const Wide other = shfl_xor(t & 2 ? pairs[0] : pairs[1], 2);
    const Wide a = t & 2 ? other : own, b = t & 2 ? own : other;  // weights 1, 2^32
    // (the bytes above q are zero, so b is when q < 2^32)
    const u64 w32 = pr.nbits > 32 ? 1ull << 32 : 0;
    const u64 mine = addmod(reduce128(a.hi, a.lo, pr), mulmod(reduce128(b.hi, b.lo, pr), w32, pr), pr.q);
    const int row = g + 8 * (t >> 1);
    if (row < nr) {
      u64* h = A.H[member] + ((size_t)(T.tile * 16 + T.ra + row - A.l0) * 2 + (t & 1)) * kN + w.x;
      *h = A.acc_in ? addmod(mine, *h, pr.q) : mine;
    }
  }
  if (!ok && lane == 0) atomicExch(A.err, 1);
}

// bytes n = 0..7 of four words, as eight words {a.n, b.n, c.n, d.n}
__device__ __forceinline__ void transpose_bytes(const u64 (&w)[4], u32 (&o)[8]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const u32 a = (u32)(w[0] >> (32 * h)), b = (u32)(w[1] >> (32 * h)), c = (u32)(w[2] >> (32 * h)),
              d = (u32)(w[3] >> (32 * h));
    const u32 ab0 = __byte_perm(a, b, 0x5140), cd0 = __byte_perm(c, d, 0x5140);
    const u32 ab2 = __byte_perm(a, b, 0x7362), cd2 = __byte_perm(c, d, 0x7362);
    o[4 * h] = __byte_perm(ab0, cd0, 0x5410);
    o[4 * h + 1] = __byte_perm(ab0, cd0, 0x7632);
    o[4 * h + 2] = __byte_perm(ab2, cd2, 0x5410);
    o[4 * h + 3] = __byte_perm(ab2, cd2, 0x7632);
  }
}

constexpr int PACK_X = 32, PACK_THREADS = 256;

// Split-format words [nl][ell][kN] of layers l0.. (within one tile) to table
// rows.  A block takes 32 points and one step: warps read runs of 32 points,
// the rows are put together in shared memory and written as runs of
// nl * 16 NPL bytes.
template <int NPL>
__global__ void __launch_bounds__(PACK_THREADS) k_pack_planes(DevView V, const u64* __restrict__ src, int ell, int l0,
                                                              int nl, u32 rows, int nks, unsigned char* out) {
  extern __shared__ u32 pk[];
  constexpr int W = 4 * NPL, ST = 16 * W + 1;  // words per row; point stride (odd: no bank conflicts)
  const u32 kN = (u32)V.k * V.N;
  const u32 x0 = blockIdx.x * PACK_X;
  const int ks = blockIdx.y, lane = threadIdx.x & 31;
  const u32 x = x0 + lane;
  for (int rt = threadIdx.x >> 5; rt < nl * 4; rt += PACK_THREADS / 32) {
    const int r = rt >> 2, t = rt & 3;
    u64 w[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = 16 * ks + 4 * t + b;
      w[b] = 0;
      if (x < kN && j < ell) w[b] = from_split(src[((size_t)r * ell + j) * kN + x], V.pr[x / V.N].split);
    }
    u32 o[8];
    transpose_bytes(w, o);
#pragma unroll
    for (int i = 0; i < NPL; ++i) pk[lane * ST + r * W + t * NPL + i] = o[i];
  }
  __syncthreads();
  const u32 tile = (u32)l0 >> 4;
  const int R = min(16, (int)rows - (int)(tile * 16)), ra = l0 & 15;
  for (int e = threadIdx.x; e < PACK_X * nl * W; e += PACK_THREADS) {
    const int p = e / (nl * W), i = e - p * (nl * W);
    if (x0 + p < kN) {
      u32* d = reinterpret_cast<u32*>(
          out + ((size_t)tile * 16 * kN * nks + ((size_t)(x0 + p) * nks + ks) * R + ra) * macp::row_bytes(NPL));
      d[i] = pk[p * ST + i];
    }
  }
}

// Reduced values [nl][ell][kN] back from the table rows.
__global__ void k_unpack_planes(int npl, const unsigned char* __restrict__ P, u32 rows, int l0, size_t count, int ell,
                                u32 kN, int nks, u64* out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const u32 x = (u32)(i % kN);
  const int j = (int)(i / kN % ell), l = l0 + (int)(i / kN / ell);
  const u32 tile = (u32)l >> 4;
  const int R = min(16, (int)rows - (int)(tile * 16));
  const unsigned char* row =
      P + ((size_t)tile * 16 * kN * nks + ((size_t)x * nks + j / 16) * R + (l & 15)) * macp::row_bytes(npl);
  u64 v = 0;
  for (int p = 0; p < npl; ++p) v |= (u64)row[((j >> 2 & 3) * npl + p) * 4 + (j & 3)] << (8 * p);
  out[i] = v;
}

// Request words [ell][2][kN] (reduced, or in the split format) of steps
// [ks0, ks0 + gridDim.y) to the byte format.
template <bool SPLIT>
__global__ void __launch_bounds__(PACK_THREADS) k_pack_request(DevView V, const u64* __restrict__ src, int ell, int nks,
                                                               int ks0, u32* __restrict__ out) {
  __shared__ u32 pk[PACK_X * 65];
  const u32 kN = (u32)V.k * V.N;
  const u32 x0 = blockIdx.x * PACK_X;
  const int ks = ks0 + blockIdx.y, lane = threadIdx.x & 31, c = (threadIdx.x >> 5) & 1, t = threadIdx.x >> 6;
  const u32 x = x0 + lane;
  u64 w[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int j = 16 * ks + 4 * t + b;
    w[b] = 0;
    if (x < kN && j < ell) {
      w[b] = src[((size_t)j * 2 + c) * kN + x];
      if (SPLIT) w[b] = from_split(w[b], V.pr[x / V.N].split);
    }
  }
  u32 o[8];
  transpose_bytes(w, o);
#pragma unroll
  for (int n = 0; n < 8; ++n) pk[lane * 65 + (n * 4 + t) * 2 + c] = o[n];
  __syncthreads();
  for (int e = threadIdx.x; e < PACK_X * 64; e += PACK_THREADS) {
    const u32 p = (u32)e >> 6, i = (u32)e & 63;
    if (x0 + p < kN) out[((size_t)(x0 + p) * nks + ks) * 64 + i] = pk[p * 65 + i];
  }
}

template <int NPL>
cudaError_t init_npl() {
  using namespace macp;
  cudaError_t e = cudaSuccess;
  for (const void* f : {(const void*)k_mac_planes<NPL, KS_ONE, false>, (const void*)k_mac_planes<NPL, KS_ONE, true>,
                        (const void*)k_mac_planes<NPL, KS_MANY, false>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)k_pack_planes<NPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             PACK_X * (64 * NPL + 1) * 4);
  return e;
}

#define PEPSI_NPL_DISPATCH(npl, F) \
  switch (npl) {                   \
    case 4: F(4); break;           \
    case 5: F(5); break;           \
    case 6: F(6); break;           \
    case 7: F(7); break;           \
    default: F(8); break;          \
  }

}  // namespace

cudaError_t mac_planes_init() {
  cudaError_t e = init_npl<4>();
  if (e == cudaSuccess) e = init_npl<5>();
  if (e == cudaSuccess) e = init_npl<6>();
  if (e == cudaSuccess) e = init_npl<7>();
  if (e == cudaSuccess) e = init_npl<8>();
  return e;
}

void launch_mac_planes(const DevView& V, int nq, const u32* const* C, const PlaneTab& P, u64* const* H, int ell, int l0,
                       int nl, int* err, cudaStream_t st, int ks0, int ks1, bool acc_in) {
  using namespace macp;
  const int nks = plane_steps(ell);
  if (ks1 < 0) ks1 = nks;
  if (nl <= 0 || nq <= 0 || ks0 >= ks1) return;
  if (nq == 3) {  // 8 consumer warps make two teams of three: 2.7 ms for 48 layers, against 1.2 + 1.0 ms
    launch_mac_planes(V, 2, C, P, H, ell, l0, nl, err, st, ks0, ks1, acc_in);
    launch_mac_planes(V, 1, C + 2, P, H + 2, ell, l0, nl, err, st, ks0, ks1, acc_in);
    return;
  }
  PlaneArgs A;
  A.P = P.p;
  A.rows = P.rows;
  A.l0 = l0;
  A.nl = nl;
  A.nks = nks;
  A.ks0 = ks0;
  A.ks1 = ks1;
  A.acc_in = acc_in ? 1 : 0;
  A.nq = nq;
  A.err = err;
  for (int q = 0; q < PEPSI_MAC_MAX_REQUESTS; ++q) {
    A.C[q] = C[std::min(q, nq - 1)];
    A.H[q] = H[std::min(q, nq - 1)];
  }
  const bool brief = ks1 - ks0 <= DRAIN;
  const int ks = nq > 1 && !brief ? KS_MANY : KS_ONE;
  const int teams = consumers(brief) / nq, sb = stage_bytes(P.npl, ks, nq);
  const int room = nq == 1 ? 160 * 1024 : SMEM_BUDGET - teams * 2 * MAX_STAGES * 8;
  A.nst = std::max(2, std::min(MAX_STAGES, room / (teams * sb)));
  const size_t smem = (size_t)teams * A.nst * (sb + 16);
  const u32 ntile = ((u32)(l0 + nl + 15) >> 4) - ((u32)l0 >> 4);
  const size_t items = (size_t)V.k * V.N * ntile;
  const unsigned grid = (unsigned)std::min<size_t>((size_t)sm_count(), (items + teams - 1) / teams);
#define GO(n)                                                                                            \
  if (brief) k_mac_planes<n, KS_ONE, true><<<grid, threads(true), smem, st>>>(V, A);                     \
  else if (nq > 1) k_mac_planes<n, KS_MANY, false><<<grid, threads(false), smem, st>>>(V, A);            \
  else k_mac_planes<n, KS_ONE, false><<<grid, threads(false), smem, st>>>(V, A)
  PEPSI_NPL_DISPATCH(P.npl, GO)
#undef GO
}

void launch_pack_planes(const DevView& V, const u64* words, int ell, int l0, int nl, const PlaneTab& P, cudaStream_t st) {
  const u32 kN = (u32)V.k * V.N;
  for (int done = 0; done < nl;) {  // one launch per tile
    const int n = std::min(nl - done, 16 - ((l0 + done) & 15));
    const dim3 grid((kN + PACK_X - 1) / PACK_X, plane_steps(ell));
    const u64* src = words + (size_t)done * ell * kN;
#define GO(np)                                                                                                     \
  k_pack_planes<np><<<grid, PACK_THREADS, PACK_X*(64 * np + 1) * 4, st>>>(V, src, ell, l0 + done, n, P.rows,        \
                                                                          plane_steps(ell), P.p)
    PEPSI_NPL_DISPATCH(P.npl, GO)
#undef GO
    done += n;
  }
}

void launch_unpack_planes(const DevView& V, const PlaneTab& P, int ell, int l0, int nl, u64* out, cudaStream_t st) {
  const u32 kN = (u32)V.k * V.N;
  const size_t count = (size_t)nl * ell * kN;
  if (!count) return;
  k_unpack_planes<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(P.npl, P.p, P.rows, l0, count, ell, kN,
                                                                   plane_steps(ell), out);
}

void launch_pack_request(const DevView& V, const u64* words, bool split, int ell, u32* C, cudaStream_t st, int ks0,
                         int ks1) {
  const int nks = plane_steps(ell);
  if (ks1 < 0) ks1 = nks;
  if (ks0 >= ks1) return;
  const u32 kN = (u32)V.k * V.N;
  const dim3 grid((kN + PACK_X - 1) / PACK_X, ks1 - ks0);
  if (split)
    k_pack_request<true><<<grid, PACK_THREADS, 0, st>>>(V, words, ell, nks, ks0, C);
  else
    k_pack_request<false><<<grid, PACK_THREADS, 0, st>>>(V, words, ell, nks, ks0, C);
}
