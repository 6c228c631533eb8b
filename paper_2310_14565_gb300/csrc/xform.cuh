// Launch shapes shared by the transform kernels.
#pragma once
#include <algorithm>
#include <type_traits>

#include "kernels.h"

// Threads of a block running the register-blocked NTT: one per two groups of 8
// elements from N = 4096 on (N = 4096, 1200 x 3 rows: 137 us with 256 threads, 147
// us with 128 or 512; N = 16384, 256 x 8 rows: 301 us with 1024, 321 us with 512).  N =
// 8192 takes 512 as the better one over the set sizes (h = 8, 526 layers: 12.28 ms an
// evaluation, 12.48 with 256; 74 layers: even), although 256 wins where much of the
// time is relinearisation of full launches (256 products: 2.37 ms, 2.44; the paper
// shape 15.91, 16.02), which the autotuner finds.
constexpr int NTT_MAX_THREADS = 1024;
inline int ntt_threads(int N) {
  return N >= 4096 ? N / 16 : std::max(32, N / 8);
}
// Threads of the kernels that give a block a chain of transforms (plaintexts,
// encryption, keys, decryption): their larger shared memory leaves room for two
// blocks per SM at most, so they take twice the threads.
inline int chain_threads(int N) { return N >= 16384 ? NTT_MAX_THREADS : std::max(32, std::min(512, N / 8)); }
// Threads of launches of a few blocks, whose time is one block's latency.
inline int latency_threads(int N) { return std::min(NTT_MAX_THREADS, std::max(32, N / 8)); }
// Threads of the hot-path transform kernels: the schedule's choice
// (DevView::nt, picked by the autotuner), else the default above.
inline int xform_threads(const DevView& V) { return V.nt > 0 ? V.nt : ntt_threads(V.N); }
// Threads of a transform launch of `rows` blocks: a launch that gives each
// block an SM of its own (the output stage, the lazy rounding) runs its
// rows with up to the largest blocks instead, which shortens each
// transform's chain of phases.
inline int xform_threads(const DevView& V, size_t rows) {
  const int base = xform_threads(V);
  const int wide = latency_threads(V.N);
  return rows <= (size_t)sm_count() && wide > base ? wide : base;
}
// A launch in the form for the context's primes and ring: f(PM, RING), as constants.
template <class F>
void in_form(const DevView& V, const F& f) {
  typedef std::bool_constant<true> yes;
  typedef std::bool_constant<false> no;
  typedef std::integral_constant<int, RING_ANY> any;
  typedef std::integral_constant<int, RING_SMALL> small;
  if (V.logN >= FUSED_LOGN)
    V.allpm ? f(yes(), any()) : f(no(), any());
  else
    V.allpm ? f(yes(), small()) : f(no(), small());
}
inline unsigned grid_for(size_t total, int threads) { return (unsigned)((total + threads - 1) / threads); }
// Let a kernel use all the dynamic shared memory a block may hold beside its static.
inline cudaError_t allow_smem(const void* f) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, f);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  return e;
}
inline cudaError_t allow_smem(std::initializer_list<const void*> fs) {
  cudaError_t e = cudaSuccess;
  for (const void* f : fs)
    if (e == cudaSuccess) e = allow_smem(f);
  return e;
}
