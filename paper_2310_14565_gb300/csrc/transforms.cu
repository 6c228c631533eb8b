// Batched transforms, and the affine step on the load of its inverse transform.
#include "kernels.h"
#include "ntt_block.cuh"
#include "xform.cuh"

namespace {

// ------------------------------------------------------------------ NTT
// Bound by the heavy multiply-add pipe and, nearly as long, the ALU: a block per
// row keeps every stage on chip, one read and one write of the row.  1200 x 4 rows
// of N = 8192 forward: 366 us with Shoup products and barriers of the whole block,
// 281 us with folding products, constant-XOR addressing and barriers of parts,
// 269 us compiled for folding alone.
// SPLIT: store the result in the split operand format of the
// multiply-accumulate (the request's forward transform).
template <bool PM, int RING, bool FWD, bool SPLIT = false>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_ntt(DevView V, const u64* __restrict__ src, u64* dst, int np, int p0, size_t src_os,
                      size_t dst_os, u32* sums) {
  extern __shared__ u64 sm[];
  const int N = V.N;
  const size_t r = blockIdx.x;
  const int pl = (int)(r % np);
  const size_t o = r / np;
  const u64* s = src + o * src_os + (size_t)pl * N;
  u64* d = dst + o * dst_os + (size_t)pl * N;
  const RowLd ld(s);
  if (FWD) {
    if (SPLIT)
      ntt_fwd_gg<PM, RING>(sm, ld, SplitSumSt(d, sums + o * dst_os + (size_t)pl * N, V.pr[p0 + pl].split), V, p0 + pl);
    else
      ntt_fwd_gg<PM, RING>(sm, ld, RowSt(d), V, p0 + pl);
  } else {
    ntt_inv_gg<PM, RING>(sm, ld, RowSt(d), V, p0 + pl);
  }
}

// out = a + z * b (NTT form, rows [groups][k][N], z as k residues), fused
// with the inverse NTT of out into coef: the block of a row computes the
// row on the transform's load and also stores it (each element is loaded
// once).  coef may alias b: a block reads its row of b before it writes
// that row of coef.
template <bool PM, int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1)
    k_axpy_intt(DevView V, const u64* __restrict__ a, const u64* __restrict__ zres, const u64* b, u64* __restrict__ out,
                u64* coef) {
  extern __shared__ u64 sm[];
  const int N = V.N;
  const size_t r = blockIdx.x;
  const int p = (int)(r % V.k);
  const DevPrime pr = V.pr[p];
  const u64 z = zres[p];
  const u64* ar = a + r * N;
  const u64* br = b + r * N;
  u64* ur = out + r * N;
  u64* cr = coef + r * N;
  ntt_inv_gg<PM, RING>(
      sm,
      [&](int x) {
        const u64 u = addmod(ar[x], mulmod(z, br[x], pr), pr.q);
        ur[x] = u;
        return u;
      },
      RowSt(cr), V, p);
}

}  // namespace

void launch_ntt(const DevView& V, bool fwd, const u64* src, u64* dst, size_t outer, int np, int p0, size_t src_os,
                size_t dst_os, cudaStream_t st, bool split_out, u32* sums) {
  const size_t rows = outer * (size_t)np;
  if (!rows) return;
  auto go = [&](auto kernel) {
    kernel<<<(unsigned)rows, xform_threads(V, rows), (size_t)V.N * sizeof(u64), st>>>(V, src, dst, np, p0, src_os, dst_os,
                                                                                    sums);
  };
  in_form(V, [&](auto pm, auto ring) {
    constexpr bool PM = decltype(pm)::value;
    constexpr int RING = decltype(ring)::value;
    if (fwd && split_out)
      go(k_ntt<PM, RING, true, true>);
    else if (fwd)
      go(k_ntt<PM, RING, true>);
    else
      go(k_ntt<PM, RING, false>);
  });
}

void launch_axpy_intt(const DevView& V, const u64* a, const u64* zres, const u64* b, u64* out, u64* coef,
                      size_t groups, cudaStream_t st) {
  const size_t rows = groups * V.k;
  if (!rows) return;
  auto go = [&](auto kernel) {
    kernel<<<(unsigned)rows, xform_threads(V, rows), (size_t)V.N * 8, st>>>(V, a, zres, b, out, coef);
  };
  in_form(V, [&](auto pm, auto ring) { go(k_axpy_intt<decltype(pm)::value, decltype(ring)::value>); });
}

cudaError_t transforms_init() {
  // (rings below 4096 stay within the default limit)
  return allow_smem({(const void*)k_ntt<true, RING_ANY, true>, (const void*)k_ntt<true, RING_ANY, false>,
                     (const void*)k_ntt<true, RING_ANY, true, true>, (const void*)k_ntt<false, RING_ANY, true>,
                     (const void*)k_ntt<false, RING_ANY, false>, (const void*)k_ntt<false, RING_ANY, true, true>,
                     (const void*)k_axpy_intt<true, RING_ANY>, (const void*)k_axpy_intt<false, RING_ANY>});
}
