// Question Contrastive Teacher Selection (section "Question Contrastive Teacher Selection",
// Eq. 1 and Eq. 2): from the text-to-vision attention maps of every language-model layer,
// for the sample's question and for the fixed reference question, the per-layer target
// distributions p^l and p_ref^l, their Jensen-Shannon divergence, and the teacher layer
// l* = argmax_l D_JS(p^l, p_ref^l).
//
// The work is one streaming read of the attention maps (hundreds of MB per sample for a
// 7B backbone), so it is HBM-bound; two launches:
//   1. qcts_colsum_kernel: Eq. 1 column sums.  One CTA sums all rows (head, question token) of one
//      (sample, layer) over a tile of 64 columns: a thread owns 8 adjacent columns (one aligned
//      16-byte load per row, whatever N is) and one of 32 row phases, with 8 rows in flight, the
//      last ones too.  The 32 partial sums per column are added in a fixed order through shared
//      memory, so results do not depend on scheduling and no global scratch, atomics or other CTAs
//      are needed.  (Clusters of 8 CTAs splitting a tile's rows and adding through distributed
//      shared memory spent that time loading nothing, and narrower loads where N is not a multiple of 8
//      had a quarter or less of the bytes in flight: 2 samples of 2880 tokens, 32 x 32 maps, 205 ->
//      175 us per call, the time the measured copy rate takes; 4 of 576: 62 -> 35 us; N = 2881: 399 -> 87 us.)
//      Samples with the most rows come first in the grid, so that the last CTAs to run
//      are short.
//   2. qcts_finish_kernel: one CTA per (sample, layer): l1 normalisation of both aggregates
//      in place and the divergence; the last CTA of each sample to finish takes the argmax
//      over layers (ties to the lower layer) and copies p^{l*}.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <memory>
#include <new>

#include "../../include/map_gb300.h"
#include "ptx.cuh"

namespace mapk {
namespace {

constexpr int kTile = 64;                       // columns per tile
constexpr int kPhases = 32;                     // threads down the rows
constexpr int kUnroll = 8;                      // rows in flight per thread
constexpr int kFinishThreads = 1024;
static_assert(kFinishThreads == 32 * 32, "a warp adds the warps' sums");
constexpr int kMaxSamples = 1024;               // samples per launch (kernel-parameter table)

struct QctsMeta {
  int b0, count;       // global index of the first sample of this launch, samples in it
  int L, H, N, m_ref;
  int32_t lens[kMaxSamples];
  int32_t order[kMaxSamples];    // samples of this launch, most rows first
  long long row0[kMaxSamples];   // first row (of N elements) of each sample's question block
};
static_assert(sizeof(QctsMeta) + 7 * sizeof(void*) <= 32764, "a kernel's parameters: at most 32764 bytes");

__device__ __forceinline__ float low_bf16(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float high_bf16(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// acc[0], acc[1] += the two columns of one 32-bit word of eight rows, added as a tree.
__device__ __forceinline__ void add_words(const uint32_t (&w)[kUnroll], float* acc) {
  static_assert(kUnroll == 8, "a tree of eight rows");
  acc[0] += ((low_bf16(w[0]) + low_bf16(w[1])) + (low_bf16(w[2]) + low_bf16(w[3]))) +
            ((low_bf16(w[4]) + low_bf16(w[5])) + (low_bf16(w[6]) + low_bf16(w[7])));
  acc[1] += ((high_bf16(w[0]) + high_bf16(w[1])) + (high_bf16(w[2]) + high_bf16(w[3]))) +
            ((high_bf16(w[4]) + high_bf16(w[5])) + (high_bf16(w[6]) + high_bf16(w[7])));
}

// acc[v] += element v of the 16-byte chunks at p, p + step, ... (n of them), kUnroll loads issued
// before their adds; the last, incomplete batch is loaded under predicates (a zero added for a
// missing row), not row by row.  A chunk that reaches outside [lo, hi), the array (only its first
// or last one can), is read element by element.
__device__ __forceinline__ void add_rows(const uint16_t* p, long long step, long long n, const uint16_t* lo,
                                         const uint16_t* hi, float* acc) {
  auto by_element = [&](const uint16_t* q) {
#pragma unroll
    for (int v = 0; v < 8; ++v)
      if (q + v >= lo && q + v < hi) acc[v] += __uint_as_float(static_cast<uint32_t>(q[v]) << 16);
  };
  if (n > 0 && p < lo) {
    by_element(p);
    p += step;
    --n;
  }
  const bool last = n > 0 && p + (n - 1) * step + 8 > hi;
  if (last) --n;
  for (long long i = 0; i < n; i += kUnroll, p += kUnroll * step) {
    uint4 x[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      x[u] = i + u < n ? __ldcs(reinterpret_cast<const uint4*>(p + u * step)) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t w0[8] = {x[0].x, x[1].x, x[2].x, x[3].x, x[4].x, x[5].x, x[6].x, x[7].x};
    const uint32_t w1[8] = {x[0].y, x[1].y, x[2].y, x[3].y, x[4].y, x[5].y, x[6].y, x[7].y};
    const uint32_t w2[8] = {x[0].z, x[1].z, x[2].z, x[3].z, x[4].z, x[5].z, x[6].z, x[7].z};
    const uint32_t w3[8] = {x[0].w, x[1].w, x[2].w, x[3].w, x[4].w, x[5].w, x[6].w, x[7].w};
    add_words(w0, acc);
    add_words(w1, acc + 2);
    add_words(w2, acc + 4);
    add_words(w3, acc + 6);
    if (i + kUnroll >= n) {                     // p: the row after the last one
      p += (n - i) * step;
      break;
    }
  }
  if (last) by_element(p);
}

// Eq. 1 for one (sample, layer, column tile): a[n] = 1/(H M) sum_{h, m} A[h, m, n] for the
// question (into a_out) and 1/(H M_ref) sum for the reference question (into aref_out).
// Grid (column tiles, L, samples).
// Rows start at any even address (N need not be a multiple of 8), so the aligned chunks of a row
// start up to 7 columns before the tile: by the same amount in every 32nd row, i.e. in all rows of
// a thread.  GROUPS = 8 chunks cover the tile when rows are aligned (N % 8 == 0 and both arrays on
// 16 bytes), 9 otherwise; the sums of columns outside the tile are dropped.
template <int GROUPS>
__global__ void __launch_bounds__(GROUPS * kPhases, 4) qcts_colsum_kernel(const __grid_constant__ QctsMeta m,
                                                               const uint16_t* __restrict__ attn,
                                                               const uint16_t* __restrict__ attn_end,
                                                               const uint16_t* __restrict__ ref,
                                                               const uint16_t* __restrict__ ref_end,
                                                               float* __restrict__ a_out,
                                                               float* __restrict__ aref_out,
                                                               int32_t* __restrict__ teacher) {
  __shared__ float part[2][kPhases][kTile];
  pdl_enter();
  const int tile = blockIdx.x, l = blockIdx.y, bl = m.order[blockIdx.z];
  const long long b = m.b0 + bl;
  const int N = m.N;
  const int cg = threadIdx.x % GROUPS, ph = threadIdx.x / GROUPS;
  const int c0 = tile * kTile;
  if (tile == 0 && l == 0 && threadIdx.x == 0) teacher[b] = 0;   // finish-kernel counter

  const long long Rq = static_cast<long long>(m.H) * m.lens[bl], Rr = static_cast<long long>(m.H) * m.m_ref;
  const long long step = static_cast<long long>(kPhases) * N;
#pragma unroll
  for (int which = 1; which >= 0; --which) {    // the reference's few rows, then the question's
    const long long R = which ? Rr : Rq;
    const uint16_t* row = which ? ref + ((b * m.L + l) * Rr + ph) * N : attn + (m.row0[bl] + l * Rq + ph) * N;
    const int s = GROUPS == 8 ? 0 : static_cast<int>((reinterpret_cast<uintptr_t>(row + c0) >> 1) & 7u);
    const int k0 = cg * 8 - s;                  // the chunk's first column, from the tile's
    float acc[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) acc[v] = 0.f;
    if (c0 + k0 < N && k0 < kTile)
      add_rows(row + c0 + k0, step, ph < R ? (R - ph + kPhases - 1) / kPhases : 0, which ? ref : attn,
               which ? ref_end : attn_end, acc);
#pragma unroll
    for (int v = 0; v < 8; ++v)
      if (GROUPS == 8 || (k0 + v >= 0 && k0 + v < kTile)) part[which][ph][k0 + v] = acc[v];
  }
  __syncthreads();
  const int Mb = m.lens[bl];
  const float scale_q = Mb > 0 ? 1.0f / (static_cast<float>(m.H) * static_cast<float>(Mb)) : 0.f;
  const float scale_r = 1.0f / (static_cast<float>(m.H) * static_cast<float>(m.m_ref));
  for (int i = threadIdx.x; i < 2 * kTile; i += GROUPS * kPhases) {
    const int which = i / kTile, c = i - which * kTile;
    float s = 0.f;
#pragma unroll
    for (int p = 0; p < kPhases; ++p) s += part[which][p][c];
    if (c0 + c < N) {
      float* out = which ? aref_out : a_out;
      out[(b * m.L + l) * N + c0 + c] = s * (which ? scale_r : scale_q);
    }
  }
}

// Deterministic block sum of two values (kFinishThreads threads): trees within and over the warps.
__device__ __forceinline__ float2 block_sum2(float x, float y, float2* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = make_float2(x, y);
  __syncthreads();
  if (threadIdx.x < 32) {
    float2 s = red[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (threadIdx.x == 0) red[kFinishThreads / 32] = s;
  }
  __syncthreads();
  const float2 r = red[kFinishThreads / 32];
  __syncthreads();   // red may be reused
  return r;
}

// phi(d) = (1 + d) ln(1 + d) + (1 - d) ln(1 - d) >= 0, so that with m = (p + q)/2 and
// d = (p - q)/(p + q):  p ln(p/m) + q ln(q/m) = m phi(d).  For |d| < 1/4 the even power
// series phi(d) = sum_k d^(2k) / (k (2k - 1)) (six terms, truncation below 1e-9 relative)
// avoids the cancellation of the two logarithms when p is close to q.
__device__ __forceinline__ float js_phi(float d) {
  const float u = d * d;
  if (u < 0.0625f) {
    return u * (1.0f + u * (1.0f / 6.0f + u * (1.0f / 15.0f + u * (1.0f / 28.0f + u * (1.0f / 45.0f + u * (1.0f / 66.0f))))));
  }
  const float a = (1.0f + d) * log1pf(d);
  const float c = (1.0f - d) > 0.f ? (1.0f - d) * log1pf(-d) : 0.f;
  return a + c;
}

__device__ __forceinline__ float js_term(float pn, float qn) {
  const float t = pn + qn;
  return t > 0.f ? 0.5f * t * js_phi((pn - qn) / t) : 0.f;
}

// One CTA per (sample, layer): p = a / sum(a) (uniform when the sum is zero) for the
// question and the reference, written in place, and js = D_JS(p, p_ref) in nats.  The last
// CTA of a sample to finish (counted in teacher[b], zeroed by the column-sum kernel) takes
// l* = argmax_l js (ties to the lower layer), writes it over the count and copies p^{l*} to
// teacher_p.  V4: N % 4 == 0 and 16-byte aligned rows (float4 accesses).
template <bool V4>
__global__ void __launch_bounds__(kFinishThreads) qcts_finish_kernel(int L, int N, int b0, float* __restrict__ p,
                                                               float* __restrict__ pref, float* __restrict__ js,
                                                               int32_t* __restrict__ teacher,
                                                               float* __restrict__ teacher_p) {
  __shared__ float2 red[kFinishThreads / 32 + 1];
  __shared__ int last;
  pdl_enter();
  const long long b = b0 + blockIdx.y;
  const long long row = b * L + blockIdx.x;
  float* a = p + row * N;
  float* r = pref + row * N;
  const float inv_n = 1.0f / static_cast<float>(N);
  float acc = 0.f;
  if (V4) {
    const int n4 = N / 4;
    float4* a4 = reinterpret_cast<float4*>(a);
    float4* r4 = reinterpret_cast<float4*>(r);
    float sa = 0.f, sr = 0.f;
    for (int i = threadIdx.x; i < n4; i += kFinishThreads) {
      const float4 x = a4[i], y = r4[i];
      sa += (x.x + x.y) + (x.z + x.w);
      sr += (y.x + y.y) + (y.z + y.w);
    }
    const float2 s = block_sum2(sa, sr, red);
    const bool ua = !(s.x > 0.f), ur = !(s.y > 0.f);
    for (int i = threadIdx.x; i < n4; i += kFinishThreads) {
      const float4 x = a4[i], y = r4[i];
      const float4 pn = ua ? make_float4(inv_n, inv_n, inv_n, inv_n)
                           : make_float4(x.x / s.x, x.y / s.x, x.z / s.x, x.w / s.x);
      const float4 qn = ur ? make_float4(inv_n, inv_n, inv_n, inv_n)
                           : make_float4(y.x / s.y, y.y / s.y, y.z / s.y, y.w / s.y);
      a4[i] = pn;
      r4[i] = qn;
      acc += (js_term(pn.x, qn.x) + js_term(pn.y, qn.y)) + (js_term(pn.z, qn.z) + js_term(pn.w, qn.w));
    }
  } else {
    float sa = 0.f, sr = 0.f;
    for (int n = threadIdx.x; n < N; n += kFinishThreads) {
      sa += a[n];
      sr += r[n];
    }
    const float2 s = block_sum2(sa, sr, red);
    const bool ua = !(s.x > 0.f), ur = !(s.y > 0.f);
    for (int n = threadIdx.x; n < N; n += kFinishThreads) {
      const float pn = ua ? inv_n : a[n] / s.x;
      const float qn = ur ? inv_n : r[n] / s.y;
      a[n] = pn;
      r[n] = qn;
      acc += js_term(pn, qn);
    }
  }
  __threadfence();   // this thread's p, p_ref writes are visible before the sample's count moves
  const float2 tot = block_sum2(acc, 0.f, red);
  if (threadIdx.x == 0) {
    js[row] = 0.5f * tot.x;
    __threadfence();
    last = atomicAdd(teacher + b, 1) == L - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ int best_l;
  if (threadIdx.x < 32) {
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    for (int l = threadIdx.x; l < L; l += 32) {
      const float v = __ldcg(js + b * L + l);
      if (v > bv) {   // l increases within a lane: a later equal value never wins
        bv = v;
        bi = l;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) {
        bv = ov;
        bi = oi;
      }
    }
    if (threadIdx.x == 0) {
      best_l = bi < L ? bi : 0;
      teacher[b] = best_l;
    }
  }
  __syncthreads();
  if (teacher_p != nullptr) {
    const float* src = p + (b * L + best_l) * N;
    for (int n = threadIdx.x; n < N; n += kFinishThreads) teacher_p[b * N + n] = __ldcg(src + n);
  }
}

template <int GROUPS>
cudaError_t launch_colsum(const QctsMeta& m, const uint16_t* attn, const uint16_t* attn_end, const uint16_t* ref,
                          const uint16_t* ref_end, float* p, float* pref, int32_t* teacher, cudaStream_t st) {
  const dim3 grid((m.N + kTile - 1) / kTile, m.L, m.count);
  return launch_k(qcts_colsum_kernel<GROUPS>, grid, dim3(GROUPS * kPhases), 0, st, m, attn, attn_end, ref, ref_end, p,
                  pref, teacher);
}

}  // namespace
}  // namespace mapk

extern "C" int map_qcts(const void* attn, const int32_t* lens, const void* attn_ref, int M_ref, int B, int L, int H,
                        int N, float* p, float* p_ref, float* js, int32_t* teacher, float* teacher_p, void* stream) {
  using namespace mapk;
  if (!attn || !lens || !attn_ref || !p || !p_ref || !js || !teacher) return MAP_EINVAL;
  if (B < 1 || L < 1 || H < 1 || N < 1 || M_ref < 1) return MAP_EINVAL;
  if (L > 65535 || (static_cast<long long>(N) + 63) / 64 > 65535) return MAP_EUNSUPPORTED;
  for (int b = 0; b < B; ++b)
    if (lens[b] < 0) return MAP_EINVAL;
  const uintptr_t ua = reinterpret_cast<uintptr_t>(attn), ur = reinterpret_cast<uintptr_t>(attn_ref);
  if ((ua | ur) & 1u) return MAP_EINVAL;
  const bool aligned = N % 8 == 0 && ((ua | ur) & 15u) == 0;
  long long rows = 0;                                          // of all question blocks
  for (int b = 0; b < B; ++b) rows += static_cast<long long>(L) * H * lens[b];
  const uint16_t* a16 = static_cast<const uint16_t*>(attn);
  const uint16_t* r16 = static_cast<const uint16_t*>(attn_ref);
  const uint16_t* a_end = a16 + rows * N;
  const uint16_t* r_end = r16 + static_cast<long long>(B) * L * H * M_ref * N;
  const bool v4 = N % 4 == 0 && ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(p_ref)) & 15u) == 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  // samples per launch: the parameter table, and at most 65535 rows of the finish grid
  const int per_launch = std::max(1, std::min(kMaxSamples, 65535 / L));
  std::unique_ptr<QctsMeta> mp(new (std::nothrow) QctsMeta);   // 16 KB, copied into the launch parameters
  if (!mp) return MAP_ENOMEM;
  QctsMeta& m = *mp;
  long long row = 0;
  for (int b0 = 0; b0 < B; b0 += per_launch) {
    m.b0 = b0;
    m.count = std::min(per_launch, B - b0);
    m.L = L;
    m.H = H;
    m.N = N;
    m.m_ref = M_ref;
    for (int i = 0; i < m.count; ++i) {
      m.lens[i] = lens[b0 + i];
      m.row0[i] = row;
      row += static_cast<long long>(L) * H * lens[b0 + i];
      m.order[i] = i;
    }
    std::stable_sort(m.order, m.order + m.count, [&](int32_t x, int32_t y) { return m.lens[x] > m.lens[y]; });
    cudaError_t e = aligned ? launch_colsum<8>(m, a16, a_end, r16, r_end, p, p_ref, teacher, st)
                            : launch_colsum<9>(m, a16, a_end, r16, r_end, p, p_ref, teacher, st);
    if (e == cudaSuccess)
      e = v4 ? launch_k(qcts_finish_kernel<true>, dim3(L, m.count), dim3(kFinishThreads), 0, st, L, N, b0, p, p_ref, js,
                        teacher, teacher_p)
             : launch_k(qcts_finish_kernel<false>, dim3(L, m.count), dim3(kFinishThreads), 0, st, L, N, b0, p,
                        p_ref, js, teacher, teacher_p);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return e == cudaErrorInvalidValue ? MAP_EINVAL : MAP_ECUDA;
    }
  }
  return MAP_OK;
}
