// Encoding, plaintexts, keys and the client's steps (Algorithms 3, 7), the response's mask and switching.
#include <cstring>

#include "kernels.h"
#include "ntt_block.cuh"
#include "rns.cuh"
#include "xform.cuh"

namespace {

// ------------------------------------------------ parallel cuckoo rounds
// One round of the client's cuckoo placement (pepsi_params.client_cuckoo =
// 1).  state: 0 placed, 1 unplaced, 2 evicted in this round; choice: the
// item's current candidate (0..2) among bins3[3u..3u+2].  claim[b] holds the
// smallest unplaced item claiming bin b (UINT32_MAX for none).
__global__ void k_ck_claim(const u32* __restrict__ bins3, const uint8_t* __restrict__ state,
                           const uint8_t* __restrict__ choice, u32 m, u32* claim) {
  const u32 u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= m || state[u] != 1) return;
  atomicMin(&claim[bins3[3 * (size_t)u + choice[u]]], u);
}
// Per bin: its winning claimant takes the first free slot, or the slot
// (evictions mod gamma) whose occupant is evicted to its next candidate.
__global__ void k_ck_resolve(u32 nbins, u32 gamma, u32* claim, int32_t* slot_item, u32* load, u32* evictions,
                             uint8_t* state, uint8_t* choice) {
  const u32 b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbins) return;
  const u32 w = claim[b];
  if (w == 0xFFFFFFFFu) return;
  claim[b] = 0xFFFFFFFFu;
  size_t c;
  if (load[b] < gamma) {
    c = (size_t)b * gamma + load[b]++;
  } else {
    c = (size_t)b * gamma + evictions[b]++ % gamma;
    const int32_t v = slot_item[c];
    state[v] = 2;
    choice[v] = (uint8_t)((choice[v] + 1) % 3);
  }
  slot_item[c] = (int32_t)w;
  state[w] = 0;
}
// Claimants that lost move to their next candidate; the evicted become
// unplaced; *unplaced counts both.
__global__ void k_ck_advance(u32 m, uint8_t* state, uint8_t* choice, u32* unplaced) {
  const u32 u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= m) return;
  if (state[u] == 1) {
    choice[u] = (uint8_t)((choice[u] + 1) % 3);
    atomicAdd(unplaced, 1u);
  } else if (state[u] == 2) {
    state[u] = 1;
    atomicAdd(unplaced, 1u);
  }
}

// ---------------------------------------------------------- CW unranking
// v = sum_{r=1..h} C(c_r, r) with c_1 < ... < c_h (combinatorial number
// system); binom[c*(h+1)+r] = C(c, r) for c <= ell.
__global__ void k_cw_unrank(const u64* __restrict__ T, size_t count, const u64* __restrict__ binom, int ell, int h,
                            uint16_t* pos) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  u64 v = T[i];
  uint16_t* o = pos + i * h;
  if (v == PEPSI_DUMMY) {
    o[0] = PEPSI_CW_NONE;
    return;
  }
  int hi = ell;  // exclusive upper bound for c_r
  for (int r = h; r >= 1; --r) {
    // largest c in [r-1, hi) with C(c, r) <= v
    int lo = r - 1, up = hi - 1;
    while (lo < up) {
      int mid = (lo + up + 1) >> 1;
      if (binom[(size_t)mid * (h + 1) + r] <= v)
        lo = mid;
      else
        up = mid - 1;
    }
    o[r - 1] = (uint16_t)lo;
    v -= binom[(size_t)lo * (h + 1) + r];
    hi = lo;
  }
}

// floor(x / t) with the one-word Barrett constant of t
__device__ __forceinline__ u64 div_by(u64 x, const DevPrime& t) {
  const u64 d = __umul64hi(x, t.m64);  // short by at most 1
  return x - d * t.q >= t.q ? d + 1 : d;
}
// round(Q m / t) mod q_p for m in [0, t): floor(Q/t) m + round((Q mod t) m / t)
__device__ __forceinline__ u64 delta_of(const RnsConst& rc, u64 m, int p, const DevPrime& pq, const DevPrime& t) {
  const u64 a = shoup(m, rc.qdt_q[p], rc.qdt_qs[p], pq.q);
  return addmod(a, barrett64(div_by(rc.qmt * m + (t.q - 1) / 2, t), pq), pq.q);
}
// sample_uniform modulo p.q, with p's reduction constants (2^64 mod q = c64) in
// place of two 64-bit remainders
__device__ __forceinline__ u64 sample_mod(u64 key, u64 pos, const DevPrime& p) {
  u64 r = 0;
  for (u64 a = 0; a < 256; a++) {
    r = draw_keyed(key, (pos << 8) | a);
    if (p.c64 == 0 || r < (u64)(0 - p.c64)) break;
  }
  return barrett64(r, p);
}
// Encode: inverse transform modulo t of ld (a slot value below t per position)
// into m[], in 32-bit words for t below 2^30.  a: N words of scratch.
template <int RING, class Load>
__device__ __forceinline__ void encode_block(u64* a, const Load& ld, u32* m, const DevView& V) {
  if (V.pr[V.tidx].q < (1ull << 30))
    ntt_inv_gg_small<RING>(reinterpret_cast<u32*>(a), ld, [&](int i, u32 v) { m[i] = v; }, V, V.tidx);
  else
    ntt_inv_gg<false, RING>(a, [&](int i) -> u64 { return ld(i); }, [&](int i, u64 v) { m[i] = (u32)v; }, V, V.tidx);
  __syncthreads();
}

// ------------------------------------------------- server plaintexts (K3)
// Block (layer l, j-chunk): bit planes of the layer's codewords, encoded
// (inverse NTT mod t of the slot vector in bit-reversed order), centred
// lift into each q_p and forward NTT; stored in the split operand format.
template <bool PM, int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_ptgen(DevView V, const uint16_t* __restrict__ pos, int ell, int h, int JC, u64* P) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k;
  const int words = N / 32 > 0 ? N / 32 : 1;
  u64* poly = sm;                                  // N u64
  u32* mbuf = reinterpret_cast<u32*>(sm + N);      // N u32
  u32* bits = mbuf + N;                            // JC * words u32
  const int l = blockIdx.y;
  const int j0 = blockIdx.x * JC;
  for (int x = threadIdx.x; x < JC * words; x += blockDim.x) bits[x] = 0;
  __syncthreads();
  const uint16_t* lp = pos + (size_t)l * N * h;
  for (int s = threadIdx.x; s < N; s += blockDim.x) {
    const uint16_t* ps = lp + (size_t)s * h;
    if (ps[0] == PEPSI_CW_NONE) continue;
    for (int r = 0; r < h; ++r) {
      int c = (int)ps[r] - j0;
      if (c >= 0 && c < JC) atomicOr(&bits[c * words + (s >> 5)], 1u << (s & 31));
    }
  }
  __syncthreads();
  const DevPrime Pt = V.pr[V.tidx];
  const u64 t = Pt.q, thalf = t >> 1;
  for (int jj = 0; jj < JC; ++jj) {
    const int j = j0 + jj;
    if (j >= ell) break;
    // Encode: slot s at position brev(s), inverse NTT mod t into mbuf
    const u32* bj = bits + jj * words;
    encode_block<RING>(
        poly,
        [&](int i) -> u32 {
          const u32 s = brev_bits(i, V.logN);
          return (bj[s >> 5] >> (s & 31)) & 1u;
        },
        mbuf, V);
    for (int p = 0; p < k; ++p) {
      // centred lift to q_p on the load, split operand format on the store
      const u64 q = V.pr[p].q, sp = V.pr[p].split;
      u64* out = P + (((size_t)l * ell + j) * k + p) * N;
      ntt_fwd_gg<PM, RING>(
          poly,
          [&](int i) -> u64 {
            const u64 m = mbuf[i];
            return m <= thalf ? m : q - (t - m);
          },
          SplitSt(out, sp), V, p);
      __syncthreads();  // the next transform overwrites poly
    }
  }
}

// Value plaintexts of labelled PSI / PSI-Sum (Algorithms 4-5): for layer
// l (one block each), slots V[l][.] -> Encode (inverse NTT mod t, slot s at
// position brev(s)) -> centred lift -> forward NTT for every prime of
// Q u B.  Out VP[l][k+kb][N] (plain residues, not the split format).
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_valgen(DevView V, const u32* __restrict__ vals, u64* VP) {
  extern __shared__ u64 sm[];
  const int N = V.N, np = V.k + V.kb;
  u64* poly = sm;                              // N u64
  u32* mbuf = reinterpret_cast<u32*>(sm + N);  // N u32
  const int l = blockIdx.x;
  const u32* row = vals + (size_t)l * N;
  for (int i = threadIdx.x; i < N; i += blockDim.x) poly[nsw(i)] = row[brev_bits(i, V.logN)];
  __syncthreads();
  ntt_inv_view(poly, V, V.tidx);
  for (int i = threadIdx.x; i < N; i += blockDim.x) mbuf[i] = (u32)poly[nsw(i)];
  __syncthreads();
  const u64 t = V.pr[V.tidx].q, thalf = t >> 1;
  for (int p = 0; p < np; ++p) {
    const u64 q = V.pr[p].q;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const u64 m = mbuf[i];
      poly[nsw(i)] = m <= thalf ? m : q - (t - m);
    }
    __syncthreads();
    ntt_fwd_view(poly, V, p);
    u64* out = VP + ((size_t)l * np + p) * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) out[i] = poly[nsw(i)];
    __syncthreads();
  }
}

// ---------------------------------------------------------------- client
__device__ __forceinline__ u64 smod_dev(i64 v, u64 q) { return v >= 0 ? (u64)v : q - (u64)(-v); }

// Block per ciphertext j: encode bit plane j, then for each prime sample
// a, compute c0 = e - a s + round(Q m / t), c1 = a (coefficient form).
template <bool PM, int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_encrypt(DevView V, const uint16_t* __restrict__ pos, int h, const u64* __restrict__ s_ntt, u64 seed,
                          u64 idx0, u64* cts) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k, j = blockIdx.x;
  u64* poly = sm;
  u32* mbuf = reinterpret_cast<u32*>(sm + N);
  const DevPrime t = V.pr[V.tidx];
  encode_block<RING>(
      poly,
      [&](int i) -> u32 {
        const uint16_t* ps = pos + (size_t)brev_bits(i, V.logN) * h;
        u32 bit = 0;
        if (ps[0] != PEPSI_CW_NONE)
          for (int r = 0; r < h; ++r) bit |= (ps[r] == j);
        return bit;
      },
      mbuf, V);
  const u64 key_e = stream_key(seed, make_stream(STREAM_ENC_E, idx0 + j, 0));
  for (int p = 0; p < k; ++p) {
    const DevPrime pq = V.pr[p];
    const u64 key_a = stream_key(seed, make_stream(STREAM_ENC_A, idx0 + j, p));
    u64* c0 = cts + (((size_t)j * 2 + 0) * k + p) * N;
    u64* c1 = cts + (((size_t)j * 2 + 1) * k + p) * N;
    const u64* sr = s_ntt + (size_t)p * N;
    // a, its transform times s left in place, and back: every thread's last
    // elements of the first transform are its first of the second
    ntt_fwd_gg<PM, RING>(
        poly,
        [&](int i) {
          const u64 a = sample_mod(key_a, i, pq);
          c1[i] = a;
          return a;
        },
        [&](int i, u64 v) { poly[nsw(i)] = mulmod(v, sr[i], pq); }, V, p);
    ntt_inv_gg<PM, RING>(
        poly, [&](int i) { return poly[nsw(i)]; },
        [&](int i, u64 v) {
          const u64 e = smod_dev(sample_cbd21(key_e, i), pq.q);
          c0[i] = addmod(submod(e, v, pq.q), delta_of(*V.rc, mbuf[i], p, pq, t), pq.q);
        },
        V, p);
    __syncthreads();  // the next transform overwrites poly
  }
}

__global__ void k_keygen_s(DevView V, u64 seed, int8_t* s) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= V.N) return;
  const u64 key = stream_key(seed, make_stream(STREAM_SK, 0, 0));
  s[n] = (int8_t)((int)sample_uniform(key, n, 3) - 1);
}
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_keygen_sntt(DevView V, const int8_t* __restrict__ s, u64* s_ntt) {
  extern __shared__ u64 sm[];
  const int p = blockIdx.x, N = V.N;
  const u64 q = V.pr[p].q;
  for (int i = threadIdx.x; i < N; i += blockDim.x) sm[nsw(i)] = smod_dev(s[i], q);
  __syncthreads();
  ntt_fwd_view(sm, V, p);
  for (int i = threadIdx.x; i < N; i += blockDim.x) s_ntt[(size_t)p * N + i] = sm[nsw(i)];
}
// Block (digit i, prime j): rlk_i = (-a_i s + e_i + g_i s^2, a_i) in NTT form,
// g_i = 1 mod q_i and 0 mod q_j for j != i.
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_keygen_rlk(DevView V, u64 seed, const u64* __restrict__ s_ntt, u64* rlk) {
  extern __shared__ u64 sm[];
  const int N = V.N, k = V.k;
  const int i = blockIdx.x / k, j = blockIdx.x % k;
  const DevPrime pj = V.pr[j];
  u64* r0 = rlk + (((size_t)i * 2 + 0) * k + j) * N;
  u64* r1 = rlk + (((size_t)i * 2 + 1) * k + j) * N;
  const u64 key_e = stream_key(seed, make_stream(STREAM_RLK_E, i, 0));
  const u64 key_a = stream_key(seed, make_stream(STREAM_RLK_A, i, j));
  for (int x = threadIdx.x; x < N; x += blockDim.x) sm[nsw(x)] = smod_dev(sample_cbd21(key_e, x), pj.q);
  __syncthreads();
  ntt_fwd_view(sm, V, j);
  for (int x = threadIdx.x; x < N; x += blockDim.x) r0[x] = sm[nsw(x)];
  __syncthreads();
  for (int x = threadIdx.x; x < N; x += blockDim.x) sm[nsw(x)] = sample_uniform(key_a, x, pj.q);
  __syncthreads();
  ntt_fwd_view(sm, V, j);
  const u64* sr = s_ntt + (size_t)j * N;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const u64 a = sm[nsw(x)], sv = sr[x];
    u64 v = submod(r0[x], mulmod(a, sv, pj), pj.q);
    if (i == j) v = addmod(v, mulmod(sv, sv, pj), pj.q);
    r0[x] = v;
    r1[x] = a;
  }
}

// Decryption, step 1: z = c0 + c1 s per prime (coefficient form).
template <int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_dec_z(DevView V, const u64* __restrict__ ct, const u64* __restrict__ s_ntt, u64* z) {
  extern __shared__ u64 sm[];
  const int p = blockIdx.x, N = V.N, k = V.k;
  const DevPrime pq = V.pr[p];
  const u64* c1 = ct + ((size_t)k + p) * N;
  const u64 *c0 = ct + (size_t)p * N, *sr = s_ntt + (size_t)p * N;
  u64* zr = z + (size_t)p * N;
  ntt_fwd_gg<false, RING>(
      sm, [&](int i) { return c1[i]; }, [&](int i, u64 v) { sm[nsw(i)] = mulmod(v, sr[i], pq); }, V, p);
  ntt_inv_gg<false, RING>(
      sm, [&](int i) { return sm[nsw(i)]; }, [&](int i, u64 v) { zr[i] = addmod(v, c0[i], pq.q); }, V, p);
}
__device__ __forceinline__ void garner_any(const RnsArgs& A, const u64* x, u64* v) {
  if (A.rc.pm)
    garner_q<0, true>(A, x, v);
  else
    garner_q<0, false>(A, x, v);
}
// Step 2, per coefficient: m = round(t z / Q) mod t exactly (Garner of
// w = t z + (Q-1)/2 over Q, then (w - [w]_Q)/Q mod t), and the noise
// |[t z]_Q| (centred) as a double, maximised over coefficients.
__global__ void k_dec_coef(const __grid_constant__ RnsArgs A, DevView V, const u64* __restrict__ z, u32* m,
                           unsigned long long* maxr) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int N = V.N, k = V.k;
  const RnsConst* rc = &A.rc;
  const DevPrime Pt = V.pr[V.tidx];
  const u64 t = Pt.q;
  double rabs = 0.0;
  if (n < N) {
    u64 w[PEPSI_MAXQ], v[PEPSI_MAXQ];
#pragma unroll
    for (int i = 0; i < PEPSI_MAXQ; ++i)
      if (i < k) {
        const u64 q = V.pr[i].q;
        w[i] = addmod(shoup(z[(size_t)i * N + n], rc->t_q[i], rc->t_qs[i], q), rc->qhalf_q[i], q);
      }
    garner_any(A, w, v);
    u64 wq = 0;
#pragma unroll
    for (int l = 0; l < PEPSI_MAXQ; ++l)
      if (l < k) wq = barrett64(wq + barrett64(v[l], Pt) * rc->pq_t[l], Pt);  // below t + (t - 1)^2 < 2^64
    m[n] = (u32)barrett64(submod(rc->qhalf_t, wq, t) * rc->qinv_t, Pt);
#pragma unroll
    for (int i = 0; i < PEPSI_MAXQ; ++i)
      if (i < k) w[i] = shoup(z[(size_t)i * N + n], rc->t_q[i], rc->t_qs[i], V.pr[i].q);
    garner_any(A, w, v);
    if (digits_greater<PEPSI_MAXQ>(v, rc->qhalf_dig, k)) {
#pragma unroll
      for (int i = 0; i < PEPSI_MAXQ; ++i)
        if (i < k) w[i] = w[i] ? V.pr[i].q - w[i] : 0;
      garner_any(A, w, v);
    }
#pragma unroll
    for (int l = 0; l < PEPSI_MAXQ; ++l)
      if (l < k) rabs += (double)v[l] * rc->pq_d[l];
  }
  // block max, then one atomic per block (positive doubles order like u64)
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) rabs = fmax(rabs, __shfl_down_sync(0xffffffffu, rabs, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = rabs;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) b = fmax(b, red[i]);
    atomicMax(maxr, (unsigned long long)__double_as_longlong(b));
  }
}
// Step 3: slots = values of m at psi_t^(2s+1): forward NTT mod t, slot s in position brev(s).
template <int RING>
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_dec_slots(DevView V, const u32* __restrict__ m, u32* slots) {
  extern __shared__ u64 sm[];
  ntt_fwd_gg<false, RING>(
      sm, [&](int i) -> u64 { return m[i]; }, [&](int i, u64 v) { slots[brev_bits(i, V.logN)] = (u32)v; }, V, V.tidx);
}

// Modulus switching of the response to the first r primes: per
// coefficient, with z = c + (Q'-1)/2, [z]_{Q'} from Garner over the dropped
// primes, y = (z - [z]_{Q'}) / Q' mod q_i = round(c~ / Q') for any
// representative c of the residue class mod Q (Q' odd, no ties).
__global__ void k_modswitch(const __grid_constant__ ModSwitchArgs M, DevView V, const u64* __restrict__ in,
                            u64* __restrict__ out, size_t n) {
  const int N = V.N, k = M.k, r = M.r, m = k - r;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // over n*2*N
  if (idx >= n * 2 * N) return;
  const int x = (int)(idx % N);
  const size_t cc = idx / N;  // ciphertext * 2 + component
  const u64* src = in + cc * k * N + x;
  u64 v[PEPSI_MAXQ];
#pragma unroll
  for (int j = 0; j < PEPSI_MAXQ; ++j) {
    if (j < m) {
      const DevPrime d = V.pr[r + j];
      u64 z = addmod(src[(size_t)(r + j) * N], M.h[r + j], d.q);
#pragma unroll
      for (int l = 0; l < PEPSI_MAXQ; ++l)
        if (l < j) z = mulmod(submod(z, barrett64(v[l], d), d.q), M.ginv[j][l], d);
      v[j] = z;
    }
  }
  u64* dst = out + cc * r * N + x;
  for (int i = 0; i < r; ++i) {
    const DevPrime qi = V.pr[i];
    u64 S = 0;
#pragma unroll
    for (int j = 0; j < PEPSI_MAXQ; ++j)
      if (j < m) S = addmod(S, mulmod(barrett64(v[j], qi), M.pw[i][j], qi), qi.q);
    dst[(size_t)i * N] = mulmod(submod(addmod(src[(size_t)i * N], M.h[i], qi.q), S, qi.q), M.qdinv[i], qi);
  }
}

// Cardinality mask (Algorithm 5): r_s uniform in Z_t for s < N-1,
// r_{N-1} = -sum; c0 += round(Q Encode(r) / t).  A block per prime: each draws
// and encodes the same mask and adds it to its row (one block for all rows, with
// 64-bit remainders, took 73 us at N = 8192, k = 4).
__global__ void __launch_bounds__(NTT_MAX_THREADS, 1) k_mask(DevView V, u64 seed, u64* ct) {
  extern __shared__ u64 sm[];
  __shared__ u64 red[32];
  const int N = V.N, p = blockIdx.x;
  u32* r = reinterpret_cast<u32*>(sm + N);
  const DevPrime t = V.pr[V.tidx], pq = V.pr[p];
  const u64 key = stream_key(seed, make_stream(STREAM_MASK, 0, 0));
  u64 part = 0;  // below N t < 2^46
  for (int s = threadIdx.x; s < N - 1; s += blockDim.x) {
    const u64 v = sample_mod(key, s, t);
    r[s] = (u32)v;
    part += v;
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    u64 sum = 0;
    for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) sum += red[i];
    sum = barrett64(sum, t);
    r[N - 1] = sum ? (u32)(t.q - sum) : 0;
  }
  __syncthreads();
  u64* row = ct + (size_t)p * N;
  auto ld = [&](int i) -> u32 { return r[brev_bits(i, V.logN)]; };
  auto st = [&](int i, u64 v) { row[i] = addmod(row[i], delta_of(*V.rc, v, p, pq, t), pq.q); };
  if (t.q < (1ull << 30))
    ntt_inv_gg_small(reinterpret_cast<u32*>(sm), ld, st, V, V.tidx);
  else
    ntt_inv_gg(sm, [&](int i) -> u64 { return ld(i); }, st, V, V.tidx);
}

}  // namespace

void launch_cuckoo_round(const u32* bins3, u32 m, u32 nbins, u32 gamma, u32* claim, int32_t* slot_item, u32* load,
                         u32* evictions, uint8_t* state, uint8_t* choice, u32* unplaced, cudaStream_t st) {
  if (!m) return;
  k_ck_claim<<<grid_for(m, 256), 256, 0, st>>>(bins3, state, choice, m, claim);
  k_ck_resolve<<<grid_for(nbins, 256), 256, 0, st>>>(nbins, gamma, claim, slot_item, load, evictions, state, choice);
  k_ck_advance<<<grid_for(m, 256), 256, 0, st>>>(m, state, choice, unplaced);
}

void launch_cw_unrank(const u64* T, size_t count, const u64* binom, int ell, int h, uint16_t* pos, cudaStream_t st) {
  if (!count) return;
  k_cw_unrank<<<grid_for(count, 256), 256, 0, st>>>(T, count, binom, ell, h, pos);
}

static int ptgen_jc(int N) { return N >= 16384 ? 8 : 32; }
static size_t ptgen_smem(int N) {
  const int words = N / 32 > 0 ? N / 32 : 1;
  return (size_t)N * 8 + (size_t)N * 4 + (size_t)ptgen_jc(N) * words * 4;
}

void launch_ptgen(const DevView& V, const uint16_t* pos, int L, int ell, int h, u64* P, cudaStream_t st) {
  if (L <= 0) return;
  const int JC = ptgen_jc(V.N);
  dim3 grid((ell + JC - 1) / JC, L);
  auto go = [&](auto kernel) { kernel<<<grid, chain_threads(V.N), ptgen_smem(V.N), st>>>(V, pos, ell, h, JC, P); };
  in_form(V, [&](auto pm, auto ring) { go(k_ptgen<decltype(pm)::value, decltype(ring)::value>); });
}

int ptgen_layers(const DevView& V, int ell) {
  const int chunks = (ell + ptgen_jc(V.N) - 1) / ptgen_jc(V.N);  // blocks of a layer
  int per_sm = 1;
  in_form(V, [&](auto pm, auto ring) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ptgen<decltype(pm)::value, decltype(ring)::value>,
                                                  chain_threads(V.N), ptgen_smem(V.N));
  });
  const int slots = std::max(1, sm_count() * per_sm);
  int best = 16;
  double use = 0;
  for (int L = 16; L <= 64; L += 16) {
    const int blocks = L * chunks, waves = (blocks + slots - 1) / slots;
    const double u = (double)blocks / ((double)waves * slots);
    if (u > use + 0.02) {
      use = u;
      best = L;
    }
  }
  return best;
}

void launch_valgen(const DevView& V, const u32* vals, int L, u64* VP, cudaStream_t st) {
  if (L <= 0) return;
  k_valgen<<<L, chain_threads(V.N), (size_t)V.N * 12, st>>>(V, vals, VP);
}

void launch_encrypt(const DevView& V, const uint16_t* pos, int ell, int h, const u64* s_ntt, u64 seed, u64 idx0,
                    u64* cts, cudaStream_t st) {
  if (ell <= 0) return;
  auto go = [&](auto kernel) {
    kernel<<<ell, chain_threads(V.N), (size_t)V.N * 12, st>>>(V, pos, h, s_ntt, seed, idx0, cts);
  };
  in_form(V, [&](auto pm, auto ring) { go(k_encrypt<decltype(pm)::value, decltype(ring)::value>); });
}

void launch_keygen(const DevView& V, u64 seed, int8_t* s, u64* s_ntt, u64* rlk, cudaStream_t st) {
  k_keygen_s<<<grid_for(V.N, 256), 256, 0, st>>>(V, seed, s);
  k_keygen_sntt<<<V.k, chain_threads(V.N), (size_t)V.N * 8, st>>>(V, s, s_ntt);
  k_keygen_rlk<<<V.k * V.k, chain_threads(V.N), (size_t)V.N * 8, st>>>(V, seed, s_ntt, rlk);
}

void launch_modswitch(const DevView& V, const ModSwitchArgs& M, const u64* in, u64* out, size_t n, cudaStream_t st) {
  const size_t total = n * 2 * V.N;
  if (!total) return;
  k_modswitch<<<grid_for(total, 256), 256, 0, st>>>(M, V, in, out, n);
}

void launch_decrypt(const DevView& V, const u64* ct, const u64* s_ntt, u64* zbuf, u32* mbuf, u32* slots,
                    unsigned long long* maxr, cudaStream_t st) {
  cudaMemsetAsync(maxr, 0, sizeof(unsigned long long), st);
  const bool small = V.logN < FUSED_LOGN;
  auto z = small ? k_dec_z<RING_SMALL> : k_dec_z<RING_ANY>;
  z<<<V.k, latency_threads(V.N), (size_t)V.N * 8, st>>>(V, ct, s_ntt, zbuf);
  k_dec_coef<<<grid_for(V.N, 128), 128, 0, st>>>(*V.host_args, V, zbuf, mbuf, maxr);
  auto to_slots = small ? k_dec_slots<RING_SMALL> : k_dec_slots<RING_ANY>;
  to_slots<<<1, latency_threads(V.N), (size_t)V.N * 8, st>>>(V, mbuf, slots);
}

void launch_mask(const DevView& V, u64 seed, u64* ct, cudaStream_t st) {
  k_mask<<<V.k, latency_threads(V.N), (size_t)V.N * 12, st>>>(V, seed, ct);
}

cudaError_t client_init(int N) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  // largest request: the plaintext generator at this N
  if ((size_t)optin < ptgen_smem(N) || (size_t)optin < (size_t)N * 12) return cudaErrorInvalidValue;
  return allow_smem({(const void*)k_ptgen<true, RING_ANY>, (const void*)k_ptgen<false, RING_ANY>,
                     (const void*)k_ptgen<true, RING_SMALL>, (const void*)k_ptgen<false, RING_SMALL>,
                     (const void*)k_valgen, (const void*)k_encrypt<true, RING_ANY>,
                     (const void*)k_encrypt<false, RING_ANY>, (const void*)k_keygen_sntt, (const void*)k_keygen_rlk,
                     (const void*)k_dec_z<RING_ANY>, (const void*)k_dec_slots<RING_ANY>, (const void*)k_mask});
}
