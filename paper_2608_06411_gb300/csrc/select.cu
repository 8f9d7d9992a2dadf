// Diversity-aware token selection, Eq. 4 (section "Inference-Time Token Pruning").
//
// The paper keeps an orthonormal basis B of the retained embeddings and picks
//   i_t = argmax_i p_hat_i * ||v_i - B B^T v_i||.
// Here B is never formed in D-space.  With G = V V^T, the coordinates of token i on the
// basis vectors are the rows of an incremental Cholesky factor:
//   e_beta[i] = (G[j_beta, i] - sum_{beta' < beta} e_beta'[j_beta] e_beta'[i]) / r_{j_beta},
//   r_i^2     = ||v_i||^2 - sum_beta e_beta[i]^2,
// where j_beta is the token that added basis vector beta and r_{j_beta} its residual at
// that time (the same quantities Gram-Schmidt would produce, in exact arithmetic).
//
// The greedy picks are sequential, but the Gram entries they need are dense products
// <v_i, v_j>, computed on the tensor cores in blocks.
//   R0     : the first K0 picks (top-K0 by p_hat) are forced, in p_hat order; their basis is
//            the Cholesky factor of G[R0, R0] (sel_chol_kernel).  A tensor-core projection
//            of every token on that basis (gemm_tc.cu; its first 128 vectors) then gives every
//            candidate its exact value (or a bound).
// Later picks proceed in rounds:
//   choose : active set A = the s candidates with the largest value bound U (a stale
//            value, or p_hat * ||v||^lambda for tokens never evaluated; values only shrink
//            as B grows, so U is always an upper bound).
//   gram   : the products of A's rows with A's and the newer basis tokens' on tcgen05 (sel_gram.cu).
//   update : bring each A member's coordinates up to date (exact values).
//   resgram: replace G[A, A] by the Gram matrix of the residuals on the current basis, so
//            that the picks need only the coordinates added during the round.
//   greedy : pick while the best exact value in A beats the largest bound outside A (theta):
//            such a pick is the exact argmax over all candidates.  Each pick updates the
//            other A members.  Values are compared as the 64-bit key (value bits, ~index),
//            i.e. value descending, ties to the lower index; they are held squared
//            (p^2 rho^(2 lambda), same order, no square root).
// The result equals the eager fp32 greedy whatever s is; s only changes how much work is
// batched.
#include <algorithm>
#include <cstring>
#include <vector>

#include "kernels.h"
#include "newton.cuh"
#include "ptx.cuh"
#include "select.h"

namespace mapk {

namespace {

__device__ __forceinline__ uint64_t make_key(float v, int idx) {
  const float c = v > 0.f ? v : 0.f;            // values are >= 0: bit order = numeric order
  return (static_cast<uint64_t>(__float_as_uint(c)) << 32) | static_cast<uint64_t>(0xFFFFFFFFu - static_cast<uint32_t>(idx));
}
__device__ __forceinline__ int key_index(uint64_t key) {
  return static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(key & 0xFFFFFFFFull));
}

// The caller's buffers: through s.uptr when set (the cached loop graph was built for another
// call's pointers), else the fields themselves.
__device__ __forceinline__ const float* sel_scores(const SelState& s) {
  return s.uptr ? static_cast<const float*>(s.uptr[0]) : s.scores;
}
__device__ __forceinline__ const void* sel_features(const SelState& s) { return s.uptr ? s.uptr[1] : s.V; }

// Selection value, squared: p^2 * rho^(2 lambda) orders candidates like p * rho^lambda (both are
// >= 0) and needs no square root for lambda = 1.  rho^2 = r2 unless r2 <= tau ||v||^2 (then 0).
__device__ __forceinline__ float sel_value(float p, float r2, float sq, float lam, float tau) {
  if (!(p > 0.f)) return 0.f;
  if (lam == 0.f) return p * p;
  if (!(r2 > tau * sq) || !(r2 > 0.f)) return 0.f;
  const float v = lam == 1.f ? (p * p) * r2 : (p * p) * powf(r2, lam);
  return v > 0.f ? v : 0.f;
}

// Two fp32 fused multiply-adds in one instruction (the halves of a 64-bit register pair).
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float sum2(uint64_t a) {
  return __uint_as_float(static_cast<uint32_t>(a)) + __uint_as_float(static_cast<uint32_t>(a >> 32));
}

// k-th largest of n distinct 64-bit keys in shared memory (1 <= k <= n), by a block of kKthThreads:
// MSB-first radix select, 11 bits per pass (the first digit is the value's exponent and three
// mantissa bits, so that values of one magnitude already part; eight bits, all but one of the exponent, left
// them together and took a pass or two more).  Two bins a thread, found by a scan over the block.  As
// soon as the bin that holds the k-th key holds no other key, that key is the answer (usually after two
// passes).  A warp whose keys all share a bin adds once, so that a common digit is no serialisation
// point.  One image of 2880 tokens, two selections a call: 246.8 -> 242.8 us; 16 of 7290: 1741 -> 1726.
constexpr int kKthThreads = 1024;
struct KthShared {
  uint32_t hist[2 * kKthThreads];
  uint32_t warp_sum[32];
  uint32_t bin, want, count;
  uint64_t found;
};
__device__ uint64_t block_kth_largest(const uint64_t* keys, int n, int k, KthShared& sh) {
  constexpr int kBits = 11;
  uint64_t prefix = 0, mask = 0;
  uint32_t want = k;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int top = 64; top > 0;) {
    const int bits = min(kBits, top), shift = top - bits;
    const uint32_t dmask = (1u << bits) - 1u;
    sh.hist[t] = 0u;
    sh.hist[kKthThreads + t] = 0u;
    __syncthreads();
    for (int i0 = 0; i0 < n; i0 += kKthThreads) {
      const int i = i0 + t;
      const bool in = i < n && (keys[i] & mask) == prefix;
      const uint32_t digit = in ? static_cast<uint32_t>(keys[i] >> shift) & dmask : 0xFFFFFFFFu;
      int same;
      __match_all_sync(0xffffffffu, digit, &same);
      if (same) {
        if (in && lane == 0) atomicAdd(&sh.hist[digit], 32u);
      } else if (in) {
        atomicAdd(&sh.hist[digit], 1u);
      }
    }
    __syncthreads();
    // thread t owns bins 2047 - 2 t and 2046 - 2 t: counts from the top
    const uint32_t c0 = sh.hist[2 * kKthThreads - 1 - 2 * t], c1 = sh.hist[2 * kKthThreads - 2 - 2 * t];
    uint32_t incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) sh.warp_sum[warp] = incl;
    __syncthreads();
    uint32_t w = lane < warp ? sh.warp_sum[lane] : 0u;
    w = __reduce_add_sync(0xffffffffu, w);
    const uint32_t before = w + incl - (c0 + c1);      // keys in higher bins than this thread's
    if (before < want && w + incl >= want) {
      const bool first = before + c0 >= want;
      sh.bin = 2 * kKthThreads - 1 - 2 * t - (first ? 0 : 1);
      sh.want = want - before - (first ? 0u : c0);
      sh.count = first ? c0 : c1;
    }
    __syncthreads();
    prefix |= static_cast<uint64_t>(sh.bin) << shift;
    mask |= static_cast<uint64_t>(dmask) << shift;
    want = sh.want;
    top = shift;
    if (sh.count == 1u && top > 0) {                   // uniform: the k-th key is the bin's only key
      for (int i = t; i < n; i += kKthThreads)
        if ((keys[i] & mask) == prefix) sh.found = keys[i];
      __syncthreads();
      return sh.found;
    }
    __syncthreads();
  }
  return prefix;
}

// Sort `cap` (a power of two) keys descending in shared memory (bitonic network).
__device__ void block_sort_desc(uint64_t* a, int cap) {
  for (int size = 2; size <= cap; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < (cap >> 1); i += blockDim.x) {
        const int lo = (i / stride) * 2 * stride + (i % stride), hi = lo + stride;
        const bool desc = (lo & size) == 0;
        const uint64_t x = a[lo], y = a[hi];
        if (desc ? (x < y) : (x > y)) { a[lo] = y; a[hi] = x; }
      }
      __syncthreads();
    }
  }
}

__device__ void block_sort_asc_i32(int32_t* a, int n, int cap) {
  for (int i = n + threadIdx.x; i < cap; i += blockDim.x) a[i] = 0x7FFFFFFF;
  __syncthreads();
  for (int size = 2; size <= cap; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < (cap >> 1); i += blockDim.x) {
        const int lo = (i / stride) * 2 * stride + (i % stride), hi = lo + stride;
        const bool asc = (lo & size) == 0;
        const int32_t x = a[lo], y = a[hi];
        if (asc ? (x > y) : (x < y)) { a[lo] = y; a[hi] = x; }
      }
      __syncthreads();
    }
  }
}

__host__ __device__ inline int pow2_at_least(int n) {
  int c = 1;
  while (c < n) c <<= 1;
  return c;
}

// ------------------------------------------------------------------ init
// U = (p_hat * ||v||^lambda)^2, r2 = ||v||^2, nothing cached; R0 = top-K0 by p_hat, in order.
__global__ void __launch_bounds__(kKthThreads) sel_init_kernel(SelState s) {
  pdl_enter();
  extern __shared__ uint64_t sh64[];
  const int b = blockIdx.x;
  const long long base = static_cast<long long>(b) * s.N;
  __shared__ KthShared kth;
  __shared__ int cnt;
  const int nv = s.nvalid ? s.nvalid[b] : s.N;
  for (int i = threadIdx.x; i < s.N; i += blockDim.x) {
    if (i >= nv) {                       // padding: never a candidate, key below every token's
      s.U[base + i] = 0.f;
      s.r2[base + i] = 0.f;
      s.cstep[base + i] = 0;
      s.state[base + i] = 2;
      sh64[i] = 0ull;
      continue;
    }
    const float p = s.scores[base + i], sq = s.sqn ? s.sqn[base + i] : 0.f;
    s.U[base + i] = sel_value(p, sq, sq, s.lambda, s.tau);
    s.r2[base + i] = sq;
    s.cstep[base + i] = 0;
    s.state[base + i] = 0;
    sh64[i] = make_key(p, i);
  }
  if (b == 0 && threadIdx.x == 0) {   // counters of this selection (earlier readers have completed)
    if (s.bcount) { s.bcount[0] = 0; s.bcount[1] = 0; }
    if (s.done_count) *s.done_count = 0;
    if (s.uptr) { s.uptr[0] = s.scores; s.uptr[1] = s.V; }
  }
  if (threadIdx.x == 0) {
    s.npicks[b] = 0; s.nbasis[b] = 0; s.done[b] = 0; s.gbase[b] = 0;
    if (s.proj_lim) s.proj_lim[b] = 0;
    cnt = 0;
  }
  __syncthreads();
  if (s.K0 > 0) {
    const uint64_t T = block_kth_largest(sh64, s.N, s.K0, kth);
    uint64_t* sel = sh64 + s.N;
    const int cap = pow2_at_least(s.K0);
    for (int i = threadIdx.x; i < s.N; i += blockDim.x)
      if (sh64[i] >= T) sel[atomicAdd(&cnt, 1)] = sh64[i];
    if (s.K0 <= static_cast<int>(blockDim.x)) {
      // The keys are distinct (each holds its token index), so a key's place in descending
      // order is the number of larger keys: one pass, no sorting network.
      __syncthreads();
      if (static_cast<int>(threadIdx.x) < s.K0) {
        const uint64_t x = sel[threadIdx.x];
        int rank = 0;
        for (int j = 0; j < s.K0; ++j) rank += sel[j] > x ? 1 : 0;
        s.r0[static_cast<long long>(b) * s.K + rank] = key_index(x);
      }
    } else {
      for (int i = s.K0 + threadIdx.x; i < cap; i += blockDim.x) sel[i] = 0ull;
      __syncthreads();
      block_sort_desc(sel, cap);
      for (int i = threadIdx.x; i < s.K0; i += blockDim.x) s.r0[static_cast<long long>(b) * s.K + i] = key_index(sel[i]);
    }
  }
}

// ------------------------------------------------------------------ choose
// Active set of the next round: the next R0 chunk (forced), else the S candidates with the
// largest bound U (value descending, ties to the lower index) and theta = the next key.
__global__ void __launch_bounds__(kKthThreads) sel_choose_kernel(SelState s) {
  pdl_enter();
  extern __shared__ uint64_t sh64[];
  const int b = blockIdx.x;
  const long long base = static_cast<long long>(b) * s.N;
  const int S = s.S;
  int32_t* aslot = s.aslot + static_cast<long long>(b) * S;
  if (s.done[b]) return;
  const int np = s.npicks[b];
  uint64_t theta = 0;
  int mode;
  if (np < s.K0) {
    const int na = min(S, s.K0 - np);
    for (int i = threadIdx.x; i < S; i += blockDim.x)
      aslot[i] = i < na ? s.r0[static_cast<long long>(b) * s.K + np + i] : -1;
    mode = 1;
  } else {
    __shared__ KthShared kth;
    __shared__ int cnt, n_alive;
    if (threadIdx.x == 0) { cnt = 0; n_alive = 0; }
    __syncthreads();
    int alive = 0;
    for (int i = threadIdx.x; i < s.N; i += blockDim.x) {
      const bool a = s.state[base + i] == 0;
      sh64[i] = a ? make_key(s.U[base + i], i) : 0ull;
      alive += a;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) alive += __shfl_xor_sync(0xffffffffu, alive, o);
    if ((threadIdx.x & 31) == 0 && alive) atomicAdd(&n_alive, alive);
    __syncthreads();
    // keys > theta form A; theta = the (S+1)-th largest key (0: nothing outside A)
    if (n_alive > S) theta = block_kth_largest(sh64, s.N, S + 1, kth);
    for (int i = threadIdx.x; i < s.N; i += blockDim.x)
      if (sh64[i] > theta) aslot[atomicAdd(&cnt, 1)] = i;
    __syncthreads();
    for (int i = cnt + threadIdx.x; i < S; i += blockDim.x) aslot[i] = -1;
    mode = 0;
  }
  if (threadIdx.x == 0) {
    s.mode[b] = mode;
    s.theta[b] = theta;
    // a projection since the last choose: later Gram blocks start past the coordinates it gave
    if (s.proj_lim && s.proj_lim[b] > 0) {
      s.gbase[b] = min(s.nbasis[b], kReprojMax);
      s.proj_lim[b] = 0;
    }
  }
}

// Sets up a projection: which images to project (first: all; otherwise those still selecting whose
// basis has grown and has at most kReprojMax vectors), their list for the projection GEMM, and the
// rows of their basis in Vg: row S + beta <- basis token beta.  kGatherCtas CTAs per image, each
// walking every kGatherCtas-th row.  proj_lim is read back by the next choose.
constexpr int kGatherCtas = 64;
constexpr int kGatherThreads = 128;

__global__ void __launch_bounds__(kGatherThreads) sel_gather_kernel(SelState s, int first) {
  pdl_enter();
  const int b = blockIdx.y;
  const bool go = first || (!s.done[b] && s.nbasis[b] > s.gbase[b] && s.nbasis[b] <= kReprojMax);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (b == 0) s.bcount[s.bc_par ^ 1] = 0;
    s.proj_lim[b] = go ? kReprojMax : 0;
    if (go) s.blist[atomicAdd(s.bcount + s.bc_par, 1)] = b;
  }
  if (!go) return;
  const int nb = min(s.nbasis[b], kReprojMax);
  const int vec = s.D / 8;
  for (int r = blockIdx.x; r < nb; r += kGatherCtas) {
    const int src = s.basis_tok[static_cast<long long>(b) * s.K + r];
    const uint4* __restrict__ V = reinterpret_cast<const uint4*>(sel_features(s)) + (static_cast<long long>(b) * s.N + src) * vec;
    uint4* __restrict__ dst = reinterpret_cast<uint4*>(s.Vg) + (static_cast<long long>(b) * s.R + s.S + r) * vec;
    // four 16-byte loads in flight per thread before their stores (V and Vg never overlap)
    int c = threadIdx.x;
    constexpr int T = kGatherThreads;
    for (; c + 3 * T < vec; c += 4 * T) {
      const uint4 x0 = __ldg(V + c), x1 = __ldg(V + c + T), x2 = __ldg(V + c + 2 * T), x3 = __ldg(V + c + 3 * T);
      dst[c] = x0;
      dst[c + T] = x1;
      dst[c + 2 * T] = x2;
      dst[c + 3 * T] = x3;
    }
    for (; c < vec; c += T) dst[c] = __ldg(V + c);
  }
}

// ------------------------------------------------------------------ coordinates
// Per-slot coordinate rows in shared memory have a pitch of 4 (mod 8) floats, so that eight
// lanes reading 16 bytes each from eight rows hit disjoint banks.
constexpr int kChunk = 32;
constexpr int kUpdSlots = 16;
constexpr int kRoundPitch = kRoundPicks + 4;

__host__ __device__ inline int coord_pitch(int KP) { return ((KP + 7) / 8) * 8 + 4; }

// ------------------------------------------------------------------ update
// Brings every active token's coordinates up to the current basis (nb vectors) by forward
// substitution before the picks:
//   e_beta[i] = (G[j_beta, i] - sum_{beta' < beta} e_beta'[j_beta] e_beta'[i]) / r_beta,
// 32 basis vectors (a chunk) at a time.  The slots are independent, the chunks are not: what
// bounds it is a chunk's latency, so a CTA serves only 16 slots (16 CTAs an image), their
// coordinate rows in shared memory.  For a chunk starting at b0 the products with the coordinates
// before it, P[slot][row] = sum_{q < b0} e_q[slot] L[row][q] (L rows: the chunk's basis tokens' own
// coordinate rows), form a 16 x 32 x b0 matrix product: each warp takes every eighth
// 16-column block with 4 slots x 4 rows per thread, then each thread adds the eight partial
// products of two entries.  Warp 0 solves the chunk's 32 x 32 triangle right-looking (lane = slot:
// each new coordinate is subtracted from the later ones at once), dividing by the basis norm as a
// product with its reciprocal and one correction step (newton.cuh: without the division's chain in every
// step), while the other warps copy the next chunk's L rows,
// triangle, Gram entries and basis norms into shared memory (cp.async), so that no chunk waits for
// a global load.  Writes Ec, r2 and cstep = nb.
// k = 640 of 2880, 2 images, a round at 560 vectors: 90 us with the triangle's 32 steps unrolled and
// branching per slot, 82 us like this.  32 slots and four warps a CTA took about twice that; 8 slots a
// CTA were slower in a batch (the L rows are copied twice as often), and a second buffer of L rows did
// not help.
constexpr int kUpdWarps = 8;

__global__ void __launch_bounds__(32 * kUpdWarps) sel_update_kernel(SelState s) {
  pdl_enter();
  extern __shared__ __align__(16) float shu[];           // [kUpdSlots][P] slot rows, then [32][P] L rows
  // a chunk's triangle by columns, LT[q][i] = L[b0 + i][b0 + q], q < i; zeros past column 31
  __shared__ __align__(16) float LT[2][kChunk][kChunk + 24];
  __shared__ float gsm[2][kUpdSlots][kChunk + 1];        // its Gram entries G[slot][b0 + i]
  __shared__ float rn[2][kChunk];                        // its basis norms
  __shared__ float part[kUpdWarps][kUpdSlots][kChunk + 1];
  static_assert(kUpdSlots * kChunk == 2 * 32 * kUpdWarps, "two entries of a chunk per thread");
  __shared__ int tok_s[kUpdSlots], c0_s[kUpdSlots];
  const int b = blockIdx.y;
  if (s.done[b]) return;
  const int S = s.S, R = s.R, KP = s.KP, P = coord_pitch(KP);
  float* Lb = shu + kUpdSlots * P;
  const int nb = s.nbasis[b], gbase = s.gbase[b];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long base = static_cast<long long>(b) * s.N;
  if (threadIdx.x < kUpdSlots) {
    const int slot = blockIdx.x * kUpdSlots + threadIdx.x;
    const int tok = slot < S ? s.aslot[static_cast<long long>(b) * S + slot] : -1;
    tok_s[threadIdx.x] = tok;
    c0_s[threadIdx.x] = tok >= 0 ? min(s.cstep[base + tok], nb) : nb;
  }
  __syncthreads();
  int cmin = nb;                                     // fewest cached coordinates over the slots
  for (int i = 0; i < kUpdSlots; ++i) cmin = min(cmin, c0_s[i]);
  if (cmin >= nb) return;                            // uniform
  const int32_t* btok_g = s.basis_tok + static_cast<long long>(b) * s.K;
  const float* rnorm = s.rnorm + static_cast<long long>(b) * s.K;
  const float* Gb = s.G + (static_cast<long long>(b) * S + blockIdx.x * kUpdSlots) * R;
  // everything chunk c needs, copied by threads t0, t0 + stride, ... (one commit group)
  auto stage = [&](int c, int buf, int t0, int stride) {
    const int nch = min(nb, c + kChunk) - c, v4 = c / 4;
    for (int e = t0; e < nch * v4; e += stride) {    // L rows, columns [0, c)
      const int row = e / v4, q = (e - row * v4) * 4;
      cp_async16(Lb + row * P + q, s.Ec + (base + __ldg(btok_g + c + row)) * KP + q);
    }
    for (int e = t0; e < nch * kChunk; e += stride) {   // the triangle: row i, columns c .. c + i - 1
      const int i = e / kChunk, q = e - i * kChunk;
      if (q < i) cp_async4(&LT[buf][q][i], s.Ec + (base + __ldg(btok_g + c + i)) * KP + c + q);
    }
    for (int e = t0; e < kUpdSlots * nch; e += stride) {   // Gram entries of the slots that need them
      const int sl = e / nch, i = e - sl * nch;
      if (tok_s[sl] >= 0 && c + i >= c0_s[sl]) cp_async4(&gsm[buf][sl][i], Gb + static_cast<long long>(sl) * R + S + c + i - gbase);
    }
    for (int e = t0; e < nch; e += stride) cp_async4(&rn[buf][e], rnorm + c + e);
    cp_async_commit();
  };
  for (int r = warp; r < kUpdSlots; r += kUpdWarps) {   // cached coordinates [0, c0) of every slot
    const int tok = tok_s[r], c0 = c0_s[r];
    if (tok < 0) continue;
    const float* g = s.Ec + (base + tok) * KP;
    float* me = shu + r * P;
    for (int q = 4 * lane; q < c0; q += 128) cp_async16(me + q, g + q);
  }
  for (int i = threadIdx.x; i < 2 * kChunk * 24; i += 32 * kUpdWarps) LT[i / (24 * kChunk)][i / 24 % kChunk][kChunk + i % 24] = 0.f;
  const int first = (cmin / kChunk) * kChunk;
  stage(first, 0, threadIdx.x, blockDim.x);
  const int mtok = lane < kUpdSlots ? tok_s[lane] : -1, mc0 = lane < kUpdSlots ? c0_s[lane] : nb;   // warp 0: this lane's slot
  float r2 = warp == 0 && mtok >= 0 ? s.r2[base + mtok] : 0.f;
  const int sg = lane >> 3, rg = lane & 7;           // products: slots 4 sg + 0..3, rows rg + 8 j
  int buf = 0;
  for (int b0 = first; b0 < nb; b0 += kChunk, buf ^= 1) {
    const int nch = min(nb, b0 + kChunk) - b0;
    cp_async_wait_all();                             // this chunk's copies (and the slot rows)
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[u][j] = 0.f;
    for (int qa = 16 * warp; qa < b0; qa += 16 * kUpdWarps) {   // whole 16-column blocks (b0 % 32 == 0)
#pragma unroll
      for (int q4 = 0; q4 < 16; q4 += 4) {
        float4 m[4], l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) m[u] = *reinterpret_cast<const float4*>(shu + (4 * sg + u) * P + qa + q4);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          l[j] = rg + 8 * j < nch ? *reinterpret_cast<const float4*>(Lb + (rg + 8 * j) * P + qa + q4)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float t = acc[u][j];
            t = fmaf(m[u].x, l[j].x, t);
            t = fmaf(m[u].y, l[j].y, t);
            t = fmaf(m[u].z, l[j].z, t);
            acc[u][j] = fmaf(m[u].w, l[j].w, t);
          }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < 4; ++j) part[warp][4 * sg + u][rg + 8 * j] = acc[u][j];
    __syncthreads();                                 // products done: Lb is free
#pragma unroll
    for (int h = 0; h < 2; ++h) {                    // a thread reads and writes its own entries only
      const int sl = warp + kUpdWarps * h;
      part[0][sl][lane] =
          gsm[buf][sl][lane] - (((part[0][sl][lane] + part[1][sl][lane]) + (part[2][sl][lane] + part[3][sl][lane])) +
                                ((part[4][sl][lane] + part[5][sl][lane]) + (part[6][sl][lane] + part[7][sl][lane])));
    }
    __syncthreads();
    if (warp != 0) {
      if (b0 + kChunk < nb) stage(b0 + kChunk, buf ^ 1, threadIdx.x - 32, blockDim.x - 32);
    } else {
      // eight basis vectors per pass, then the row shifts down by eight: the code stays small, and
      // without branches (a slot without a token, a cached coordinate, a vector past nb are selects)
      const float my_rn = lane < nch ? rn[buf][lane] : 1.f, my_inv = lane < nch ? 1.0f / my_rn : 0.f;
      const bool act = mtok >= 0;
      float* me = shu + (lane & (kUpdSlots - 1)) * P + b0;
      float av[kChunk];
#pragma unroll
      for (int i = 0; i < kChunk; ++i) av[i] = part[0][lane & (kUpdSlots - 1)][i];
#pragma unroll 1
      for (int t0 = 0; t0 < nch; t0 += 8) {
        float old[8], ev[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) old[u] = t0 + u < nch ? me[t0 + u] : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float ri = __shfl_sync(0xffffffffu, my_inv, t0 + u), rr = __shfl_sync(0xffffffffu, my_rn, t0 + u);
          const bool fresh = b0 + t0 + u >= mc0 && t0 + u < nch;   // past nb: e = 0
          const float e = fresh ? quotient(av[u], rr, ri) : old[u];
          r2 = fresh ? fmaf(-e, e, r2) : r2;
          ev[u] = e;
#pragma unroll
          for (int j = (u + 1) & ~3; j < kChunk; j += 4) {
            const float4 l = *reinterpret_cast<const float4*>(&LT[buf][t0 + u][t0 + j]);
            if (j > u) av[j] = fmaf(-e, l.x, av[j]);
            if (j + 1 > u) av[j + 1] = fmaf(-e, l.y, av[j + 1]);
            if (j + 2 > u) av[j + 2] = fmaf(-e, l.z, av[j + 2]);
            if (j + 3 > u) av[j + 3] = fmaf(-e, l.w, av[j + 3]);
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (act && t0 + u < nch) me[t0 + u] = ev[u];
#pragma unroll
        for (int j = 0; j < 24; ++j) av[j] = av[j + 8];
#pragma unroll
        for (int j = 24; j < 32; ++j) av[j] = 0.f;
      }
    }
    __syncthreads();                                 // this chunk's coordinates are written
  }
  if (warp == 0 && mtok >= 0 && mc0 < nb) {
    s.r2[base + mtok] = r2;
    s.cstep[base + mtok] = nb;
  }
  for (int r = warp; r < kUpdSlots; r += kUpdWarps) {   // new coordinates [c0, nb), a warp per row
    const int tok = tok_s[r], c0 = c0_s[r];
    if (tok < 0 || c0 >= nb) continue;
    float* g = s.Ec + (base + tok) * KP;
    const float* me = shu + r * P;
    for (int q = c0 + lane; q < nb; q += 32) g[q] = me[q];
  }
}

// ------------------------------------------------------------------ R0 basis
// The K0 forced picks (R0 in p_hat order) need no argmax: their basis is the Cholesky factor
// of the K0 x K0 Gram matrix G[R0, R0] in pick order.  Column t adds a basis vector unless its
// residual is degenerate (r^2 <= tau ||v||^2: the column is zero and is dropped when the
// coordinates are written); its entries below the diagonal are the later R0 tokens'
// coordinates.  Writes picks, state, basis, Ec rows, cstep and r2 of the R0 tokens.
//
// Blocked, 32 columns (a panel) at a time, so that only the 32 x 32 diagonal block is a
// sequential chain, and that one stays inside a warp (a barrier and a whole dot product per
// column made up nearly all of the column-by-column form's time):
//   1. the panel less its products with the columns before it, a register-tiled matrix product;
//   2. the diagonal block by warp 0, lane = row, the row in registers, shuffles for the others';
//   3. the rows below it, a thread per row, by forward substitution against the block.
// One image, K0 = 80: 35.4 -> 23.0 us; 16 images, K0 = 202: 70.5 us for 128 columns and a forced
// round for the rest -> 77.6 us for all of them (ncu, cold).
// In shared memory, rows of panel b hold 32 (b + 1) columns and 4 of padding: eight consecutive
// rows read 16 bytes each from 32 different banks.
constexpr int kCholThreads = 256;
static_assert(kCholMax <= kCholThreads && kCholMax % 32 == 0, "a thread per R0 token");

// First float of row u in the panel-wise lower triangle.
__host__ __device__ inline int chol_row(int u) {
  const int p = u / 32;
  return 32 * (16 * p * (p + 1) + 4 * p) + (u - 32 * p) * (32 * (p + 1) + 4);
}

__global__ void __launch_bounds__(kCholThreads, 1) sel_chol_kernel(SelState s) {
  pdl_enter();
  extern __shared__ __align__(16) float A[];           // G, then L, in place
  // the diagonal block's columns: LT[t][j] = L[c0 + j][c0 + t], zero for j <= t and past 31
  __shared__ __align__(16) float LT[32][56];
  __shared__ float rinv_s[32];                         // 1 / r of its columns, 0: no basis vector
  __shared__ float dg[kCholMax], dpick[kCholMax];
  __shared__ int tk[kCholMax], mine_s[kCholMax], ext_s[kCholMax];
  const int b = blockIdx.x, K0 = s.K0;
  const int npan = (K0 + 31) / 32;
  const long long base = static_cast<long long>(b) * s.N;
  const float* Gb = s.G + static_cast<long long>(b) * s.S * s.R;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = warp; r < 32 * npan; r += kCholThreads / 32) {
    float* row = A + chol_row(r);
    const int w4 = 8 * (r / 32 + 1);                   // G rows are 16-byte aligned (R % 16 == 0)
    for (int c = lane; c < w4; c += 32) {
      // columns past K0 (rows too) are zero: they never extend the basis
      if (r < K0 && 4 * c + 4 <= K0) cp_async16(row + 4 * c, Gb + static_cast<long long>(r) * s.R + 4 * c);
      else
        for (int k = 0; k < 4; ++k)
          row[4 * c + k] = r < K0 && 4 * c + k < K0 ? Gb[static_cast<long long>(r) * s.R + 4 * c + k] : 0.f;
    }
  }
  for (int i = threadIdx.x; i < 32 * 24; i += kCholThreads) LT[i / 24][32 + i % 24] = 0.f;
  const int u = threadIdx.x;
  float pscore = 0.f;
  if (u < K0) {
    tk[u] = s.r0[static_cast<long long>(b) * s.K + u];
    pscore = sel_scores(s)[base + tk[u]];
  }
  cp_async_wait_all();
  __syncthreads();
  if (u < K0) dg[u] = A[chol_row(u) + u];
  else if (u < kCholMax) dg[u] = 0.f;
  __syncthreads();
  int nb = 0;                                          // basis vectors so far (warp 0)
  const int cg = threadIdx.x & 7, rg = threadIdx.x >> 3;   // products: columns cg + 8 k, row rg of each panel
  for (int pan = 0; pan < npan; ++pan) {
    const int c0 = 32 * pan;
    if (c0 > 0) {
      const float* lc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) lc[k] = A + chol_row(c0 + cg + 8 * k);
      for (int i0 = pan; i0 < npan; i0 += 4) {         // up to four row panels at a time
        float* lr[4];
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          lr[i] = A + chol_row(32 * min(i0 + i, npan - 1) + rg);
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[i][k] = 0.f;
        }
        for (int q = 0; q < c0; q += 4) {
          float4 y[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) y[k] = *reinterpret_cast<const float4*>(lc[k] + q);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (i0 + i < npan) {                       // uniform
              const float4 x = *reinterpret_cast<const float4*>(lr[i] + q);
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float v = acc[i][k];
                v = fmaf(x.x, y[k].x, v);
                v = fmaf(x.y, y[k].y, v);
                v = fmaf(x.z, y[k].z, v);
                acc[i][k] = fmaf(x.w, y[k].w, v);
              }
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i0 + i < npan) {
#pragma unroll
            for (int k = 0; k < 4; ++k) lr[i][c0 + cg + 8 * k] -= acc[i][k];
          }
      }
      __syncthreads();
    }
    if (warp == 0) {                                   // the diagonal block
      // eight columns per pass, then the row shifts down by eight: the loop's code stays small
      float a[32];
      float* row = A + chol_row(c0 + lane) + c0;
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(row + j);
        a[j] = v.x; a[j + 1] = v.y; a[j + 2] = v.z; a[j + 3] = v.w;
      }
      const float floor2 = s.tau * dg[c0 + lane];
      float mydiag = 0.f;
      bool myext = false;
      const int cols = min(32, K0 - c0);               // the last panel's other columns are empty
#pragma unroll 1
      for (int t0 = 0; t0 < cols; t0 += 8) {
        float ev[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const bool me = lane == t0 + t;
          const float d = __shfl_sync(0xffffffffu, a[t], t0 + t);
          const float fl = __shfl_sync(0xffffffffu, floor2, t0 + t);
          const bool ext = d > fl && d > 0.f;
          const float rinv = ext ? inv_sqrt(d) : 0.f;
          const float e = ext && lane > t0 + t ? a[t] * rinv : 0.f;
          if (me) { mydiag = d; myext = ext; rinv_s[t0 + t] = rinv; }
          ev[t] = e;
          LT[t0 + t][lane] = e;
          const int done = t < 7 ? t + 1 : t;          // columns up to here are up to date
          if (t < 7) a[t + 1] = fmaf(-e, __shfl_sync(0xffffffffu, e, t0 + t + 1), a[t + 1]);   // the next pivot column
          __syncwarp();
#pragma unroll
          for (int j = (done + 1) & ~3; j < 32; j += 4) {   // zero at and before column t, and past 31
            const float4 l = *reinterpret_cast<const float4*>(&LT[t0 + t][t0 + j]);
            if (j > done) a[j] = fmaf(-e, l.x, a[j]);
            if (j + 1 > done) a[j + 1] = fmaf(-e, l.y, a[j + 1]);
            if (j + 2 > done) a[j + 2] = fmaf(-e, l.z, a[j + 2]);
            if (j + 3 > done) a[j + 3] = fmaf(-e, l.w, a[j + 3]);
          }
        }
        *reinterpret_cast<float4*>(row + t0) = make_float4(ev[0], ev[1], ev[2], ev[3]);
        *reinterpret_cast<float4*>(row + t0 + 4) = make_float4(ev[4], ev[5], ev[6], ev[7]);
#pragma unroll
        for (int j = 0; j < 24; ++j) a[j] = a[j + 8];
#pragma unroll
        for (int j = 24; j < 32; ++j) a[j] = 0.f;
      }
      const unsigned m = __ballot_sync(0xffffffffu, myext);
      dpick[c0 + lane] = mydiag;
      ext_s[c0 + lane] = myext;
      mine_s[c0 + lane] = nb + __popc(m & ((1u << lane) - 1u));
      nb += __popc(m);
    }
    __syncthreads();
    const int r = c0 + 32 + threadIdx.x;               // the rows below
    if (r < K0) {
      float x[32];
      float* row = A + chol_row(r) + c0;
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(row + j);
        x[j] = v.x; x[j + 1] = v.y; x[j + 2] = v.z; x[j + 3] = v.w;
      }
#pragma unroll 1
      for (int t0 = 0; t0 < 32; t0 += 8) {
        float ev[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const float ri = rinv_s[t0 + t];
          const float e = ri != 0.f ? x[t] * ri : 0.f;
          ev[t] = e;
#pragma unroll
          for (int j = (t + 1) & ~3; j < 32; j += 4) {
            const float4 l = *reinterpret_cast<const float4*>(&LT[t0 + t][t0 + j]);
            if (j > t) x[j] = fmaf(-e, l.x, x[j]);
            if (j + 1 > t) x[j + 1] = fmaf(-e, l.y, x[j + 1]);
            if (j + 2 > t) x[j + 2] = fmaf(-e, l.z, x[j + 2]);
            if (j + 3 > t) x[j + 3] = fmaf(-e, l.w, x[j + 3]);
          }
        }
        *reinterpret_cast<float4*>(row + t0) = make_float4(ev[0], ev[1], ev[2], ev[3]);
        *reinterpret_cast<float4*>(row + t0 + 4) = make_float4(ev[4], ev[5], ev[6], ev[7]);
#pragma unroll
        for (int j = 0; j < 24; ++j) x[j] = x[j + 8];
#pragma unroll
        for (int j = 24; j < 32; ++j) x[j] = 0.f;
      }
    }
    __syncthreads();
  }
  if (u < K0) {
    const int tok = tk[u];
    const float d = dpick[u];
    s.picks[static_cast<long long>(b) * s.K + u] = tok;
    s.state[base + tok] = 1;
    s.cstep[base + tok] = mine_s[u];
    s.r2[base + tok] = d;
    s.U[base + tok] = sel_value(pscore, d, dg[u], s.lambda, s.tau);
    if (ext_s[u]) {
      s.basis_tok[static_cast<long long>(b) * s.K + mine_s[u]] = tok;
      s.rnorm[static_cast<long long>(b) * s.K + mine_s[u]] = sqrtf(d);
    }
  }
  // coordinate rows of the R0 tokens: e_beta for beta < (basis size at their pick)
  for (int r = warp; r < K0; r += kCholThreads / 32) {
    const float* row = A + chol_row(r);
    float* g = s.Ec + (base + tk[r]) * s.KP;
    for (int q = lane; q < r; q += 32)
      if (ext_s[q]) g[mine_s[q]] = row[q];
  }
  if (threadIdx.x == 0) {
    s.nbasis[b] = nb;
    s.npicks[b] = K0;
  }
}

// ------------------------------------------------------------------ residual Gram
// When a round's picks start, every active token's coordinates are current on the c0 basis
// vectors of the round (sel_update_kernel).  Over that basis the residual Gram matrix of
// the active set is
//   G'[i][k] = <v_i, v_k> - sum_{q < c0} e_q[i] e_q[k]   (the inner product of the residuals),
// and a pick then needs only the coordinates added during the round (sel_greedy_kernel).
// It replaces the lower triangle of the A x A part of the Gram block in place (no more of it is
// computed or read).  One CTA of 64 threads per 32 x 32 tile, 4 x 4 outputs per thread; the coordinates are staged in 16-column chunks,
// transposed, in two shared buffers, the next chunk loaded during the products of the
// current one.  Small tiles keep several CTAs on every SM, so the chunk loop's latency is
// hidden, with few images (c0 is large) as with many.
constexpr int kRgTile = 32, kRgChunk = 16, kRgPad = kRgTile + 4, kRgThreads = 64;

__global__ void __launch_bounds__(kRgThreads) sel_resgram_kernel(SelState s) {
  pdl_enter();
  // two buffers of both operands' chunks; after the products, the output tile
  __shared__ __align__(16) float sbuf[4 * kRgChunk * kRgPad];
  static_assert(4 * kRgChunk * kRgPad >= kRgTile * (kRgTile + 1), "tile staging");
  float(*Ei)[kRgChunk][kRgPad] = reinterpret_cast<float(*)[kRgChunk][kRgPad]>(sbuf);
  float(*Ek)[kRgChunk][kRgPad] = reinterpret_cast<float(*)[kRgChunk][kRgPad]>(sbuf + 2 * kRgChunk * kRgPad);
  __shared__ int toki[kRgTile], tokk[kRgTile];
  const int b = blockIdx.y;
  if (s.done[b]) return;
  const int c0 = s.nbasis[b];
  if (c0 == 0) return;
  const int S = s.S, KP = s.KP;
  int t = blockIdx.x, ti = 0;
  const int T = S / kRgTile;
  while (t >= T - ti) { t -= T - ti; ++ti; }
  const int tk = ti, tr = ti + t;                    // column tile, row tile (at or below the diagonal)
  const int32_t* aslot = s.aslot + static_cast<long long>(b) * S;
  const int tid = threadIdx.x;
  if (tid < kRgTile) toki[tid] = aslot[tr * kRgTile + tid];
  else tokk[tid - kRgTile] = aslot[tk * kRgTile + tid - kRgTile];
  // a tile whose rows or columns are all empty slots writes nothing
  const bool any_i = __syncthreads_or(tid < kRgTile && toki[tid] >= 0);
  const bool any_k = __syncthreads_or(tid < kRgTile && tokk[tid] >= 0);
  if (!any_i || !any_k) return;
  const long long base = static_cast<long long>(b) * s.N;
  // staging: threads 0-31 the rows of the tile's row slots, 32-63 those of its column slots
  const int lr = tid & (kRgTile - 1);
  const int ltok = tid < kRgTile ? toki[lr] : tokk[lr];
  const float* row = ltok >= 0 ? s.Ec + (base + ltok) * KP : nullptr;
  float(*Eop)[kRgChunk][kRgPad] = tid < kRgTile ? Ei : Ek;
  auto load16 = [&](int q, float* x) {
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = 0.f;
    if (!row) return;
    if (q + 16 <= c0) {
#pragma unroll
      for (int j = 0; j < 16; j += 4) {
        const float4 u = *reinterpret_cast<const float4*>(row + q + j);
        x[j] = u.x; x[j + 1] = u.y; x[j + 2] = u.z; x[j + 3] = u.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (q + j < c0) x[j] = row[q + j];
    }
  };
  const int tx = tid & 7, ty = tid >> 3;             // outputs: rows ty*4 .. +3, columns tx*4 .. +3
  float acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
  float x[16];
  load16(0, x);
  int buf = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) Eop[0][j][lr] = x[j];
  __syncthreads();
  for (int q0 = 0; q0 < c0; q0 += kRgChunk, buf ^= 1) {
    const bool more = q0 + kRgChunk < c0;
    if (more) load16(q0 + kRgChunk, x);              // next chunk in flight during the products
#pragma unroll
    for (int q = 0; q < kRgChunk; ++q) {
      const float4 a = *reinterpret_cast<const float4*>(&Ei[buf][q][ty * 4]);
      const float4 c = *reinterpret_cast<const float4*>(&Ek[buf][q][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) acc[r][cc] = fmaf(av[r], cv[cc], acc[r][cc]);
    }
    if (more) {                                      // the other buffer was last read a chunk ago
#pragma unroll
      for (int j = 0; j < 16; ++j) Eop[buf ^ 1][j][lr] = x[j];
    }
    __syncthreads();
  }
  // G' = G - acc through a shared tile, in whole rows (coalesced)
  float(*Tt)[kRgTile + 1] = reinterpret_cast<float(*)[kRgTile + 1]>(sbuf);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) Tt[ty * 4 + r][tx * 4 + cc] = acc[r][cc];
  __syncthreads();
  constexpr int kRowsPer = kRgTile * kRgTile / kRgThreads;   // rows of the tile per thread
  const int c = tid & (kRgTile - 1), r0 = tid / kRgTile;
  const bool okc = tokk[c] >= 0;
  float* g0 = s.G + (static_cast<long long>(b) * S + tr * kRgTile) * s.R + tk * kRgTile + c;
  float gv[kRowsPer];                                // every load in flight before the stores
#pragma unroll
  for (int m = 0; m < kRowsPer; ++m) {
    const int r = r0 + m * (kRgThreads / kRgTile);
    gv[m] = okc && toki[r] >= 0 ? g0[static_cast<long long>(r) * s.R] : 0.f;
  }
#pragma unroll
  for (int m = 0; m < kRowsPer; ++m) {
    const int r = r0 + m * (kRgThreads / kRgTile);
    if (okc && toki[r] >= 0) g0[static_cast<long long>(r) * s.R] = gv[m] - Tt[r][c];
  }
}

// ------------------------------------------------------------------ greedy
// One CTA of S threads per image; thread = active slot.  The lower triangle of the A x A part of
// the Gram block holds the residual Gram matrix G' on the c0 basis vectors of the round (above),
// so a pick of slot j updates slot i with the coordinates added in this launch only:
//   e_new[i] = (G'[j][i] - sum_{c0 <= q < nb} e_q[j] e_q[i]) / r_j.
// The picks are sequential, so a pick's latency is what counts; everything on its chain is on
// chip.  G' sits in shared memory, its rows padded to 16 bytes.  A slot keeps its own round
// coordinates in registers, moved there eight at a time, and in a shared row that the others
// read by 16-byte broadcasts when it wins; the residual it publishes becomes the winner's 1 / r
// beside the dot product.  The picks take one block barrier each: the winning slot is carried in
// the low bits of the key, and after the barrier a step writes no row and no residual that it reads of
// another slot (only the remaining candidates write theirs).  At most kRoundPicks picks per launch (the next round continues):
// the triangle leaves room for 88 coordinates a slot.  Bound by the chain of dependent
// instructions of a pick (two reductions of keys, the barrier, the dot product: about 930 cycles,
// 0.45 us; two slots a thread were slower, 1860 cycles, as were a branch per eight coordinates,
// 1020, and G' read from global memory).  One image, 80 picks: 80.9 -> 52.9 us; 64 images: 82.1 ->
// 52.4 us (ncu, cold).
constexpr int kRoundChunks = kRoundPicks / 8;
constexpr int kGreedyWarps = kActiveSlots / 32;
static_assert(kRoundPicks % 8 == 0 && kRoundPitch % 4 == 0, "coordinate rows in 16-byte units");
static_assert((kGreedyWarps & (kGreedyWarps - 1)) == 0, "lanes read the warps' keys round robin");

// First float of row i of the lower triangle whose rows are padded to 16 bytes.
__host__ __device__ inline int tri_row(int i) {
  const int g = i >> 2;
  return 8 * g * (g + 1) + (i & 3) * 4 * (g + 1);
}

__global__ void __launch_bounds__(kActiveSlots, 1) sel_greedy_kernel(SelState s) {
  pdl_enter();
  extern __shared__ __align__(16) float shf[];
  __shared__ uint2 wkey[2][kGreedyWarps];            // (value bits, (0xFFFF - token, slot)) per warp
  const int b = blockIdx.x;
  if (s.done[b]) return;
  constexpr int S = kActiveSlots;
  const int R = s.R, KP = s.KP;
  float* Gt = shf;                                   // [tri_row(S)] residual Gram matrix, lower triangle
  float* Er = Gt + tri_row(S);                       // [S][kRoundPitch] round coordinates
  float* pub = Er + S * kRoundPitch;                 // [S] residual^2, or -1: degenerate, no basis vector
  int32_t* tks = reinterpret_cast<int32_t*>(pub + S);   // [S] tokens of the slots
  int32_t* ends = tks + S;                           // [S] round coordinates of the slots at the end
  int32_t* pk_tok = ends + S;                        // [kRoundPicks] this launch's picks
  float* pk_r2 = reinterpret_cast<float*>(pk_tok + kRoundPicks);  // their residuals (-1: no basis vector)
  const long long base = static_cast<long long>(b) * s.N;
  const int slot = threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* Gb = s.G + static_cast<long long>(b) * S * R;
  const int tok = s.aslot[static_cast<long long>(b) * S + slot];
#pragma unroll 4
  for (int r = warp; r < S; r += kGreedyWarps) {     // padded rows, a warp per row (R % 16 == 0)
    const float* g = Gb + static_cast<long long>(r) * R + 4 * lane;
    float* d = Gt + tri_row(r) + 4 * lane;
    if (4 * lane <= r) cp_async16(d, g);
    if (4 * lane + 128 <= r) cp_async16(d + 128, g + 128);
  }
  int nb = s.nbasis[b], np = s.npicks[b];
  const int c0 = nb, np0 = np;
  const bool forced = s.mode[b] == 1;
  const uint64_t theta = s.theta[b];                 // the best key outside the active set
  const uint32_t th_v = static_cast<uint32_t>(theta >> 32);
  const uint32_t th_t = theta ? 0xFFFFu - static_cast<uint32_t>(key_index(theta)) : 0u;
  float* me = Er + slot * kRoundPitch;

  float r2 = 0.f, sq = 0.f, p = 0.f, val = 0.f;
  int mine = nb;                                     // valid coordinates at the end
  bool alive = false;
  if (tok >= 0) {
    p = sel_scores(s)[base + tok];
    alive = s.state[base + tok] == 0;
    if (s.cstep[base + tok] < nb) {                  // sel_update_kernel did not run
      atomicOr(s.status, ST_INTERNAL);
      alive = false;
    }
    r2 = s.r2[base + tok];
    sq = s.sqn[base + tok];
    val = sel_value(p, r2, sq, s.lambda, s.tau);
  }
  {
    // zero rows: the dot products read a winner's row up to the next multiple of 8
    float4* row4 = reinterpret_cast<float4*>(me);
    for (int q = 0; q < kRoundPitch / 4; ++q) row4[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  tks[slot] = tok;
  // sel_value with what does not change between picks taken out of the loop.  A slot that is not a
  // candidate (any more) goes through the same steps with a value of zero and the lowest key.
  const bool lam1 = s.lambda == 1.f;
  const float floor2 = fmaxf(s.tau * sq, 0.f);
  float pv = alive && p > 0.f ? p : 0.f;             // p_hat of a candidate
  float r2_end = r2, val_end = val;                  // residual and value of a slot that leaves
  pub[slot] = r2 > floor2 ? r2 : -1.f;
  uint32_t vkey = alive ? __float_as_uint(val) : 0u;   // val >= 0: bit order = numeric order
  uint32_t lkey = alive ? ((0xFFFFu - static_cast<uint32_t>(tok)) << 16) | static_cast<uint32_t>(slot) : 0u;
  uint64_t er[kRoundChunks][4];                      // own round coordinates, whole chunks of eight (pairs)
#pragma unroll
  for (int c = 0; c < kRoundChunks; ++c)
#pragma unroll
    for (int u = 0; u < 4; ++u) er[c][u] = 0ull;
  cp_async_wait_all();
  __syncthreads();

  int nr = 0, cc = 0;                                // round coordinates so far, whole chunks (uniform)
  const int steps = min(s.K - np, kRoundPicks);
  int step = 0;
  for (; step < steps; ++step) {
    {
      const uint32_t vm = __reduce_max_sync(0xffffffffu, vkey);
      const uint32_t lm = __reduce_max_sync(0xffffffffu, vkey == vm ? lkey : 0u);
      if (lane == 0) wkey[step & 1][warp] = make_uint2(vm, lm);
    }
    __syncthreads();
    int jslot;
    if (forced) {
      jslot = step;
      if (jslot >= S || tks[jslot] < 0) break;
    } else {
      const uint2 k = wkey[step & 1][lane & (kGreedyWarps - 1)];
      const uint32_t vm = __reduce_max_sync(0xffffffffu, k.x);
      const uint32_t lm = __reduce_max_sync(0xffffffffu, k.x == vm ? k.y : 0u);
      // nothing left, or a token outside the set may come first (uniform)
      if (lm == 0u || vm < th_v || (vm == th_v && (lm >> 16) <= th_t)) break;
      jslot = static_cast<int>(lm & 0xFFFFu);
    }
    const float r2j = pub[jslot];
    if (slot == jslot) {                             // global writes wait for the end
      alive = false;
      pv = 0.f;
      vkey = 0u;
      lkey = 0u;
      r2_end = r2;
      val_end = val;
      mine = nb + nr;
      pk_tok[step] = tok;
      pk_r2[step] = r2j >= 0.f ? r2j : -1.f;
    }
    if (r2j >= 0.f) {                                // uniform: the pick adds a basis vector
      const float gji = Gt[tri_row(max(slot, jslot)) + min(slot, jslot)];
      const ulonglong2* cj = reinterpret_cast<const ulonglong2*>(Er + jslot * kRoundPitch);
      const ulonglong2* mj = reinterpret_cast<const ulonglong2*>(me) + 2 * cc;
      // the chunk being filled, from both rows (zeros past the end; cc < kRoundChunks here)
      const ulonglong2 x0 = cj[2 * cc], x1 = cj[2 * cc + 1], m0 = mj[0], m1 = mj[1];
      const float rinv = inv_sqrt(r2j);
      uint64_t a0 = fma2(x0.x, m0.x, 0ull), a1 = fma2(x0.y, m0.y, 0ull);
      uint64_t a2 = fma2(x1.x, m1.x, 0ull), a3 = fma2(x1.y, m1.y, 0ull);
      // whole chunks, four at a time with all their loads in flight (both sides are zero at and past
      // chunk cc: one branch per 32 coordinates instead of one per eight)
#pragma unroll
      for (int g = 0; g < kRoundChunks; g += 4) {
        if (g >= cc) break;                          // uniform
        ulonglong2 x[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (g + c / 2 < kRoundChunks) x[c] = cj[2 * g + c];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (g + c < kRoundChunks) {
            a0 = fma2(x[2 * c].x, er[g + c][0], a0);
            a1 = fma2(x[2 * c].y, er[g + c][1], a1);
            a2 = fma2(x[2 * c + 1].x, er[g + c][2], a2);
            a3 = fma2(x[2 * c + 1].y, er[g + c][3], a3);
          }
      }
      const float e = (gji - ((sum2(a0) + sum2(a1)) + (sum2(a2) + sum2(a3)))) * rinv;
      r2 = fmaf(-e, e, r2);
      const bool pos = r2 > floor2;                  // floor2 >= 0: the basis can be extended
      // Candidates only: the other warps may still read the winner's residual and row in this step (one
      // barrier a pick), and its new residual, about zero, would read as degenerate.
      if (alive) {
        me[nr] = e;
        pub[slot] = pos ? r2 : -1.f;
      }
      if (lam1) val = pos ? fmaxf((pv * pv) * r2, 0.f) : 0.f;
      else val = sel_value(pv, r2, sq, s.lambda, s.tau);
      vkey = __float_as_uint(val);
      ++nr;
      if ((nr & 7) == 0) {                           // uniform: the chunk is full
        const ulonglong2 n0 = mj[0], n1 = mj[1];
#pragma unroll
        for (int c = 0; c < kRoundChunks; ++c)
          if (c == cc) { er[c][0] = n0.x; er[c][1] = n0.y; er[c][2] = n1.x; er[c][3] = n1.y; }
        ++cc;
      }
    }
  }
  np += step;
  nb += nr;
  // write back: this launch's picks, then the active tokens
  __syncthreads();
  if (threadIdx.x == 0) {
    int nbw = c0;
    for (int i = 0; i < np - np0; ++i) {
      if (pk_r2[i] >= 0.f) {
        s.basis_tok[static_cast<long long>(b) * s.K + nbw] = pk_tok[i];
        s.rnorm[static_cast<long long>(b) * s.K + nbw] = sqrtf(pk_r2[i]);
        ++nbw;
      }
    }
  }
  for (int i = threadIdx.x; i < np - np0; i += blockDim.x) {
    s.picks[static_cast<long long>(b) * s.K + np0 + i] = pk_tok[i];
    s.state[base + pk_tok[i]] = 1;
  }
  if (tok >= 0) {
    if (alive) mine = nb;
    s.cstep[base + tok] = mine;
    s.r2[base + tok] = alive ? r2 : r2_end;
    s.U[base + tok] = alive ? val : val_end;
  }
  // coordinates [c0, mine) of every slot: its round row, one warp per row
  ends[slot] = tok >= 0 ? mine : c0;
  __syncthreads();
  for (int r = warp; r < S; r += kGreedyWarps) {
    const int t = tks[r], end = ends[r];
    if (t < 0) continue;
    float* g = s.Ec + (base + t) * KP;
    const float* src = Er + r * kRoundPitch;
    for (int q = c0 + lane; q < end; q += 32) g[q] = src[q - c0];
  }
  if (threadIdx.x == 0) {
    s.nbasis[b] = nb;
    s.npicks[b] = np;
    if (np >= s.K) { s.done[b] = 1; atomicAdd(s.done_count, 1); }
  }
}

// ------------------------------------------------------------------ outputs
// keep = picks sorted ascending; pick_order = picks.
__global__ void sel_finalize_kernel(const int32_t* picks, int K, int32_t* keep, int32_t* order) {
  pdl_enter();
  extern __shared__ int32_t sh32[];
  const int b = blockIdx.x;
  const int32_t* p = picks + static_cast<long long>(b) * K;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    sh32[i] = p[i];
    if (order) order[static_cast<long long>(b) * K + i] = p[i];
  }
  __syncthreads();
  if (K <= static_cast<int>(blockDim.x)) {
    // place = number of smaller picks (equal ones, which a valid selection never has, by position)
    const int i = threadIdx.x;
    if (i < K) {
      const int32_t x = sh32[i];
      int rank = 0;
      for (int j = 0; j < K; ++j) {
        const int32_t y = sh32[j];
        rank += (y < x || (y == x && j < i)) ? 1 : 0;
      }
      keep[static_cast<long long>(b) * K + rank] = x;
    }
    return;
  }
  block_sort_asc_i32(sh32, K, pow2_at_least(K));
  for (int i = threadIdx.x; i < K; i += blockDim.x) keep[static_cast<long long>(b) * K + i] = sh32[i];
}

// The same and the compaction in one launch: a CTA per pick places it (the number of smaller picks),
// writes it to keep there and copies its row.  Bound by latency for one image, where it saves a launch and
// has the row in flight while the picks are counted: a whole call on one image of 576 tokens 152.3 -> 149.6 us,
// of 2880 tokens (k = 160) 243.3 -> 239.2 us; 16 images with k = 405 1743.9 -> 1737.9 us, 64 images with
// k = 160 2043.7 and 2043.5 us.  A pick outside the image (after a selection that a device-side error
// ended early) is reported and its row left alone, as in map_gather.
constexpr int kFinGatherThreads = 128;
__global__ void __launch_bounds__(kFinGatherThreads) sel_finalize_gather_kernel(const int32_t* __restrict__ picks, int K,
                                                                               const uint4* __restrict__ V, int N,
                                                                               int vec_per_row, int32_t* keep,
                                                                               uint4* __restrict__ out, int* status) {
  __shared__ int part[kFinGatherThreads / 32];
  pdl_enter();
  const long long b = blockIdx.y;
  const int j = blockIdx.x, tid = threadIdx.x;
  const int32_t* p = picks + b * K;
  const int32_t x = p[j];
  const bool in = x >= 0 && x < N;
  const int nvec = in ? vec_per_row : 0;
  const uint4* s = V + (b * N + (in ? x : 0)) * vec_per_row;
  uint4 first[4];                                      // the row's first loads go with the picks'
#pragma unroll
  for (int u = 0; u < 4; ++u) first[u] = tid + u * kFinGatherThreads < nvec ? __ldg(s + tid + u * kFinGatherThreads) : make_uint4(0u, 0u, 0u, 0u);
  int less = 0;
  for (int i = tid; i < K; i += kFinGatherThreads) {
    const int32_t y = p[i];
    less += (y < x || (y == x && i < j)) ? 1 : 0;
  }
  less = __reduce_add_sync(0xffffffffu, less);
  if ((tid & 31) == 0) part[tid >> 5] = less;
  __syncthreads();
  int rank = 0;
#pragma unroll
  for (int w = 0; w < kFinGatherThreads / 32; ++w) rank += part[w];
  if (tid == 0) {
    keep[b * K + rank] = x;
    if (!in) atomicOr(status, ST_BADINDEX);
  }
  uint4* d = out + (b * K + rank) * vec_per_row;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (tid + u * kFinGatherThreads < nvec) d[tid + u * kFinGatherThreads] = first[u];
  for (int v = tid + 4 * kFinGatherThreads; v < nvec; v += kFinGatherThreads) d[v] = __ldg(s + v);
}

// top-K by p_hat (lambda = 0 or K0 = K): R0 computed by sel_init is the whole answer.
__global__ void sel_copy_r0_kernel(const int32_t* r0, int K, int32_t* picks) {
  pdl_enter();
  const int b = blockIdx.x;
  for (int i = threadIdx.x; i < K; i += blockDim.x)
    picks[static_cast<long long>(b) * K + i] = r0[static_cast<long long>(b) * K + i];
}

__global__ void sel_identity_kernel(int N, int32_t* keep, int32_t* order) {
  pdl_enter();
  const int b = blockIdx.x;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    keep[static_cast<long long>(b) * N + i] = i;
    if (order) order[static_cast<long long>(b) * N + i] = i;
  }
}


// ------------------------------------------------------------------ device-side round loop
// First node of the loop graph: the WHILE body runs only if an image still selects.
__global__ void sel_loop_init_kernel(SelState s, cudaGraphConditionalHandle h, int32_t* iters) {
  if (threadIdx.x == 0) {
    *iters = 0;
    cudaGraphSetConditional(h, (*s.done_count < s.B && *s.status == 0) ? 1u : 0u);
  }
}

// Last node of the WHILE body: run another round while an image still selects, no kernel
// has reported an error and the iteration cap has not been reached (then ST_INTERNAL).
__global__ void sel_loop_cond_kernel(SelState s, cudaGraphConditionalHandle h, int32_t* iters, int cap_iters,
                                     long long* iters_total) {
  if (threadIdx.x == 0) {
    const int it = *iters + 1;
    *iters = it;
    *iters_total += 1;
    const bool pending = *s.done_count < s.B, err = *s.status != 0;
    if (pending && !err && it >= cap_iters) atomicOr(s.status, ST_INTERNAL);
    cudaGraphSetConditional(h, (pending && !err && it < cap_iters) ? 1u : 0u);
  }
}

}  // namespace

size_t sel_init_smem(int N, int K0) { return (static_cast<size_t>(N) + pow2_at_least(std::max(K0, 1))) * 8; }
size_t sel_choose_smem(int N) { return static_cast<size_t>(N) * 8; }
size_t sel_greedy_smem(int S) {
  return static_cast<size_t>(tri_row(S)) * 4 + static_cast<size_t>(S) * kRoundPitch * 4 +
         static_cast<size_t>(S) * 12 + static_cast<size_t>(kRoundPicks) * 8;
}
size_t sel_chol_smem(int K0) {
  return static_cast<size_t>(chol_row((K0 + 31) / 32 * 32)) * 4;
}
size_t sel_update_smem(int KP) {
  return static_cast<size_t>(kUpdSlots + kChunk) * coord_pitch(KP) * 4;
}

cudaError_t launch_sel_init(const SelState& s, cudaStream_t st) {
  const size_t sm = sel_init_smem(s.N, s.K0);
  cudaError_t e = cudaFuncSetAttribute(sel_init_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  return launch_k(sel_init_kernel, dim3(s.B), dim3(kKthThreads), sm, st, s);
}

cudaError_t launch_sel_choose(const SelState& s, cudaStream_t st) {
  const size_t sm = sel_choose_smem(s.N);
  cudaError_t e = cudaFuncSetAttribute(sel_choose_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  return launch_k(sel_choose_kernel, dim3(s.B), dim3(kKthThreads), sm, st, s);
}

cudaError_t launch_sel_greedy(const SelState& s, bool update, cudaStream_t st) {
  if (s.S != kActiveSlots) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (update) {
    const size_t um = sel_update_smem(s.KP);
    e = cudaFuncSetAttribute(sel_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(um));
    if (e != cudaSuccess) return e;
    e = launch_k(sel_update_kernel, dim3((s.S + kUpdSlots - 1) / kUpdSlots, s.B), dim3(32 * kUpdWarps), um, st, s);
    if (e != cudaSuccess) return e;
  }
  const int T = s.S / kRgTile;
  e = launch_k(sel_resgram_kernel, dim3(T * (T + 1) / 2, s.B), dim3(kRgThreads), 0, st, s);
  if (e != cudaSuccess) return e;
  const size_t sm = sel_greedy_smem(s.S);
  e = cudaFuncSetAttribute(sel_greedy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  return launch_k(sel_greedy_kernel, dim3(s.B), dim3(s.S), sm, st, s);
}

cudaError_t launch_sel_chol(const SelState& s, cudaStream_t st) {
  if (s.K0 < 1 || s.K0 > kCholMax || s.K0 > s.S) return cudaErrorInvalidValue;
  const size_t sm = sel_chol_smem(s.K0);
  cudaError_t e = cudaFuncSetAttribute(sel_chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  return launch_k(sel_chol_kernel, dim3(s.B), dim3(kCholThreads), sm, st, s);
}

cudaError_t launch_sel_finalize(const int32_t* picks, int B, int K, int32_t* keep, int32_t* order, cudaStream_t st) {
  const size_t sm = static_cast<size_t>(pow2_at_least(K)) * 4;
  return launch_k(sel_finalize_kernel, dim3(B), dim3(1024), sm, st, picks, K, keep, order);
}

cudaError_t launch_sel_finalize_gather(const int32_t* picks, int B, int K, const void* V, int N, int D, int32_t* keep,
                                       void* out, int* status, cudaStream_t st) {
  return launch_k(sel_finalize_gather_kernel, dim3(K, B), dim3(kFinGatherThreads), 0, st, picks, K,
                  static_cast<const uint4*>(V), N, D / 8, keep, static_cast<uint4*>(out), status);
}

cudaError_t launch_sel_copy_r0(const int32_t* r0, int B, int K, int32_t* picks, cudaStream_t st) {
  return launch_k(sel_copy_r0_kernel, dim3(B), dim3(256), 0, st, r0, K, picks);
}

cudaError_t launch_sel_gather(const SelState& s, bool first, cudaStream_t st) {
  return launch_k(sel_gather_kernel, dim3(kGatherCtas, s.B), dim3(kGatherThreads), 0, st, s, first ? 1 : 0);
}

cudaError_t launch_sel_identity(int B, int N, int32_t* keep, int32_t* order, cudaStream_t st) {
  return launch_k(sel_identity_kernel, dim3(B), dim3(256), 0, st, N, keep, order);
}

// ------------------------------------------------------------------ loop graph cache
struct SelLoopEntry {
  std::vector<long long> key;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

struct SelLoopCache {
  std::vector<SelLoopEntry> entries;   // most recently used last
  cudaStream_t cap = nullptr;          // stream the loop body is captured on
};

namespace {
constexpr size_t kSelLoopCacheMax = 8;

void release_entry(SelLoopEntry& e) {
  if (e.exec) cudaGraphExecDestroy(e.exec);
  if (e.graph) cudaGraphDestroy(e.graph);
  e.exec = nullptr;
  e.graph = nullptr;
}

long long fbits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return static_cast<long long>(u);
}
long long pbits(const void* p) { return static_cast<long long>(reinterpret_cast<uintptr_t>(p)); }

// Everything the captured kernels depend on, except the caller's scores and features (read
// through s.uptr).
std::vector<long long> loop_key(const SelState& s, long long wait_ns, int cap_iters, const int32_t* iters,
                                const long long* iters_total) {
  return {s.B, s.N, s.D, s.K, s.K0, s.S, s.R, s.KP, fbits(s.lambda), fbits(s.tau), pbits(s.sqn), pbits(s.U),
          pbits(s.r2), pbits(s.cstep), pbits(s.state), pbits(s.Ec), pbits(s.picks), pbits(s.r0), pbits(s.basis_tok),
          pbits(s.rnorm), pbits(s.npicks), pbits(s.nbasis), pbits(s.done), pbits(s.mode), pbits(s.gbase), pbits(s.proj_lim),
          pbits(s.theta), pbits(s.aslot), pbits(s.G), pbits(s.done_count), pbits(s.status), pbits(s.nvalid),
          pbits(s.uptr), wait_ns, cap_iters, pbits(iters), pbits(iters_total)};
}

// Builds the graph: [test kernel] -> WHILE { choose, Gram, update + residual Gram + greedy; test }.
cudaError_t build_loop(SelLoopCache* c, const SelState& s, long long wait_ns, int cap_iters, int32_t* iters,
                       long long* iters_total, SelLoopEntry& out) {
  cudaError_t e = cudaSuccess;
  if (!c->cap && (e = cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking)) != cudaSuccess) return e;
  cudaGraph_t g = nullptr;
  if ((e = cudaGraphCreate(&g, 0)) != cudaSuccess) return e;
  auto fail = [&](cudaError_t err) {
    cudaGraphDestroy(g);
    return err;
  };
  cudaGraphConditionalHandle h;
  if ((e = cudaGraphConditionalHandleCreate(&h, g, 0, 0)) != cudaSuccess) return fail(e);
  SelState sc = s;
  void* init_args[] = {&sc, &h, &iters};
  cudaKernelNodeParams kp = {};
  kp.func = reinterpret_cast<void*>(sel_loop_init_kernel);
  kp.gridDim = dim3(1);
  kp.blockDim = dim3(32);
  kp.kernelParams = init_args;
  cudaGraphNode_t init_node;
  if ((e = cudaGraphAddKernelNode(&init_node, g, nullptr, 0, &kp)) != cudaSuccess) return fail(e);
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t loop_node;
  if ((e = cudaGraphAddNode(&loop_node, g, &init_node, nullptr, 1, &cp)) != cudaSuccess) return fail(e);
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  if ((e = cudaStreamBeginCaptureToGraph(c->cap, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed)) !=
      cudaSuccess)
    return fail(e);
  pdl_disabled() = true;
  SelState r = s;
  if ((e = launch_sel_choose(r, c->cap)) == cudaSuccess &&
      (e = launch_sel_gram(r, r.S, r.K, wait_ns, c->cap)) == cudaSuccess)
    e = launch_sel_greedy(r, true, c->cap);
  if (e == cudaSuccess) e = launch_k(sel_loop_cond_kernel, dim3(1), dim3(32), 0, c->cap, r, h, iters, cap_iters, iters_total);
  pdl_disabled() = false;
  cudaGraph_t captured = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(c->cap, &captured);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return fail(e);
  cudaGraphExec_t x = nullptr;
  if ((e = cudaGraphInstantiate(&x, g, 0)) != cudaSuccess) return fail(e);
  out.graph = g;
  out.exec = x;
  return cudaSuccess;
}
}  // namespace

SelLoopCache* sel_loop_cache_create() { return new SelLoopCache(); }

void sel_loop_cache_destroy(SelLoopCache* c) {
  if (!c) return;
  for (auto& e : c->entries) release_entry(e);
  if (c->cap) cudaStreamDestroy(c->cap);
  delete c;
}

cudaError_t launch_sel_loop(SelLoopCache* c, const SelState& s, long long wait_ns, int cap_iters, int32_t* iters,
                            long long* iters_total, cudaStream_t st) {
  if (!c || !s.uptr || !s.done_count || !iters || !iters_total) return cudaErrorInvalidValue;
  std::vector<long long> key = loop_key(s, wait_ns, cap_iters, iters, iters_total);
  size_t hit = c->entries.size();
  for (size_t i = 0; i < c->entries.size(); ++i)
    if (c->entries[i].key == key) { hit = i; break; }
  if (hit == c->entries.size()) {
    SelLoopEntry ent;
    ent.key = std::move(key);
    const cudaError_t e = build_loop(c, s, wait_ns, cap_iters, iters, iters_total, ent);
    if (e != cudaSuccess) return e;
    if (c->entries.size() >= kSelLoopCacheMax) {
      release_entry(c->entries.front());
      c->entries.erase(c->entries.begin());
    }
    c->entries.push_back(std::move(ent));
  } else if (hit + 1 != c->entries.size()) {
    SelLoopEntry ent = std::move(c->entries[hit]);
    c->entries.erase(c->entries.begin() + static_cast<long>(hit));
    c->entries.push_back(std::move(ent));
  }
  return cudaGraphLaunch(c->entries.back().exec, st);
}

}  // namespace mapk
