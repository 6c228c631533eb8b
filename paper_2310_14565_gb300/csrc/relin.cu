// Relinearisation by RNS digits.
#include "kernels.h"
#include "ntt_block.cuh"
#include "xform.cuh"

namespace {

// The relinearisation transforms come in two register budgets: MT = 256 for
// blocks of at most 256 threads, three per SM (80 registers a thread and no spills;
// at N = 8192 with 256-thread blocks the relinearisation took 1.98 ms against
// 2.07 ms at 64), and MT = NTT_MAX_THREADS for larger blocks (64 registers; the sum on
// the inverse's load spills 332 bytes).  N <= 4096 and the schedules that take 256
// threads (the autotuner's at the paper shape) run the first; the default at N = 8192
// is 512 threads (xform.cuh).
constexpr int relin_min_blocks(int MT) { return MT <= 256 ? 3 : 1; }

// ---------------------------------------------------------- relinearise
// Bound by the heavy multiply-add pipe (256 ciphertexts of N = 8192, k = 4, both
// phases: 0.77 ms with folding products).
// Phase 1, block per row of DG[L][k+2][k][N]: row (l, i, j) holds
// NTT_{q_j}([d2]_{q_i}) for digits i < k, and NTT_{q_j}(d0), NTT_{q_j}(d1)
// for i = k, k+1.
template <int MT, bool PM, int RING>
__global__ void __launch_bounds__(MT, relin_min_blocks(MT)) k_relin_ntt(DevView V, const u64* __restrict__ D, u64* __restrict__ DG) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k;
  const size_t r = blockIdx.x;
  const int j = (int)(r % k);
  const int i = (int)((r / k) % (k + 2));
  const size_t l = r / ((size_t)k * (k + 2));
  const DevPrime pj = V.pr[j];
  const u64* row = i < k ? D + ((l * 3 + 2) * k + i) * N : D + ((l * 3 + (i - k)) * k + j) * N;
  u64* out = DG + r * N;
  ntt_fwd_gg<PM, RING>(
      sm,
      [&](int x) {
        const u64 w = row[x];
        return w >= pj.q ? barrett64(w, pj) : w;
      },
      RowSt(out), V, j);
}
// Phase 2, thread per (l, j, n): R_c = NTT(d_c) + sum_i NTT(d_i) * rlk_i[c],
// 128-bit lazy sums, one Barrett reduction per output.
__global__ void k_relin_mac(DevView V, const u64* __restrict__ DG, const u64* __restrict__ rlk, u64* __restrict__ R,
                            int L) {
  const int N = V.N, k = V.k;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // over L*k*N
  if (idx >= (size_t)L * k * N) return;
  const int n = (int)(idx % N);
  const int j = (int)((idx / N) % k);
  const size_t l = idx / ((size_t)k * N);
  const DevPrime pj = V.pr[j];
  const u64* g = DG + l * (k + 2) * k * N + (size_t)j * N + n;
  const size_t gs = (size_t)k * N;
  u64 lo0 = g[(size_t)k * gs], hi0 = 0, lo1 = g[(size_t)(k + 1) * gs], hi1 = 0;
  for (int i = 0; i < k; ++i) {
    const u64 d = g[(size_t)i * gs];
    mac128(lo0, hi0, d, __ldg(rlk + (((size_t)i * 2 + 0) * k + j) * N + n));
    mac128(lo1, hi1, d, __ldg(rlk + (((size_t)i * 2 + 1) * k + j) * N + n));
  }
  u64* o = R + ((l * 2) * k + j) * N + n;
  o[0] = reduce128(hi0, lo0, pj);
  o[(size_t)k * N] = reduce128(hi1, lo1, pj);
}

// Relinearisation fused with the affine step after it: the block of row
// (l, c, p) of U[L][2][k][N] computes R_c = NTT(d_c) + sum_i NTT(d_i) *
// rlk_i[c] (the digit rows DG of k_relin_ntt, 128-bit sums, one reduction)
// and u = R_c + z * H on the load of the inverse NTT of U, stores u and the
// coefficient-form row.  The same words as k_relin_mac followed by
// k_axpy_intt, without R in memory.
template <int MT, bool PM, int RING>
__global__ void __launch_bounds__(MT, relin_min_blocks(MT))
    k_relin_axpy_intt(DevView V, const u64* __restrict__ DG, const u64* __restrict__ rlk,
                      const u64* __restrict__ zres, const u64* __restrict__ H, u64* __restrict__ out, u64* coef) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k;
  const size_t r = blockIdx.x;
  const int p = (int)(r % k);
  const int c = (int)((r / k) % 2);
  const size_t l = r / ((size_t)2 * k);
  const DevPrime pr = V.pr[p];
  const u64 z = zres[p];
  const u64 zc = PM ? mulmod(z, 1ull << pr.s, pr) : 0;  // companion of z
  const size_t gs = (size_t)k * N;  // digit row stride
  const u64* g = DG + l * (k + 2) * gs + (size_t)p * N;
  const u64* key = rlk + ((size_t)c * k + p) * N;  // rlk_i[c] at prime p: key + i * 2 * gs
  const u64* hr = H + r * N;
  u64* ur = out + r * N;
  ntt_inv_gg<PM, RING>(
      sm,
      [&](int x) {
        u64 lo = g[(size_t)(k + c) * gs + x], hi = 0;
        for (int i = 0; i < k; ++i) mac128(lo, hi, g[(size_t)i * gs + x], __ldg(key + (size_t)i * 2 * gs + x));
        u64 u;
        if constexpr (PM) {  // z h below 2 q joins the sum before its reduction
          const u64 zh = PmMul(pr).mul(hr[x], z, zc);
          lo += zh;
          hi += lo < zh;
          u = pm_reduce(hi, lo, PmMul(pr), (int)pr.nbits);
        } else {
          u = addmod(reduce128(hi, lo, pr), mulmod(z, hr[x], pr), pr.q);
        }
        ur[x] = u;
        return u;
      },
      RowSt(coef + r * N), V, p);
}

}  // namespace

void launch_relin_digits(const DevView& V, const u64* D, u64* DG, int L, cudaStream_t st) {
  if (L <= 0) return;
  const size_t rows = (size_t)L * (V.k + 2) * V.k;
  const int nt = xform_threads(V, rows);
  auto go = [&](auto kernel) { kernel<<<(unsigned)rows, nt, (size_t)V.N * 8, st>>>(V, D, DG); };
  in_form(V, [&](auto pm, auto ring) {
    constexpr bool PM = decltype(pm)::value;
    constexpr int RING = decltype(ring)::value;
    if (nt <= 256)
      go(k_relin_ntt<256, PM, RING>);
    else
      go(k_relin_ntt<NTT_MAX_THREADS, PM, RING>);
  });
}

void launch_relin(const DevView& V, const u64* D, const u64* rlk, u64* DG, u64* R, int L, cudaStream_t st) {
  if (L <= 0) return;
  launch_relin_digits(V, D, DG, L, st);
  k_relin_mac<<<grid_for((size_t)L * V.k * V.N, 256), 256, 0, st>>>(V, DG, rlk, R, L);
}

void launch_relin_axpy_intt(const DevView& V, const u64* DG, const u64* rlk, const u64* zres, const u64* H, u64* out,
                            u64* coef, int L, cudaStream_t st) {
  const size_t rows = (size_t)L * 2 * V.k;
  if (!rows) return;
  const int nt = xform_threads(V, rows);
  auto go = [&](auto kernel) {
    kernel<<<(unsigned)rows, nt, (size_t)V.N * 8, st>>>(V, DG, rlk, zres, H, out, coef);
  };
  in_form(V, [&](auto pm, auto ring) {
    constexpr bool PM = decltype(pm)::value;
    constexpr int RING = decltype(ring)::value;
    if (nt <= 256)
      go(k_relin_axpy_intt<256, PM, RING>);
    else
      go(k_relin_axpy_intt<NTT_MAX_THREADS, PM, RING>);
  });
}

cudaError_t relin_init() {
  return allow_smem({(const void*)k_relin_ntt<256, true, RING_ANY>,
                     (const void*)k_relin_ntt<NTT_MAX_THREADS, true, RING_ANY>,
                     (const void*)k_relin_axpy_intt<256, true, RING_ANY>,
                     (const void*)k_relin_axpy_intt<NTT_MAX_THREADS, true, RING_ANY>,
                     (const void*)k_relin_ntt<256, false, RING_ANY>,
                     (const void*)k_relin_ntt<NTT_MAX_THREADS, false, RING_ANY>,
                     (const void*)k_relin_axpy_intt<256, false, RING_ANY>,
                     (const void*)k_relin_axpy_intt<NTT_MAX_THREADS, false, RING_ANY>});
}
