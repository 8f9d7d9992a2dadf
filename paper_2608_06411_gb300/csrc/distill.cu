// Predictor distillation step (section "Cross-Modal Attention Distillation"): the batch loss
// mean_b D_KL(p*_b || p_hat_b) of Eq. 3's prediction against the teacher distribution that
// QCTS selected, and its gradient with respect to every predictor weight (the backward pass
// through Eq. 3's softmax-mean, RoPE, the projections and both MLPs).
//
// Activations and gradients are fp32 (the bf16 features and weights are decoded exactly): the
// gradient is checked against a float64 oracle.  The contractions run on the tcgen05 GEMM of
// gemm_tc.cu with split-bf16 operands: an fp32 operand x is staged as three bf16 terms hi, mid,
// lo (x to about 24 significant bits), a bf16 feature or weight as itself, and the product is
// formed from every term pair above 2^-24 (six for two fp32 operands, three against an exact
// bf16 one, one for two bf16 ones), accumulated in fp32 in TMEM.  Every matrix is staged once, in
// the elementwise kernel that makes it (bias and GELU, GELU', RoPE, softmax backward; the bias
// gradients' column sums beside it), and read by every contraction that uses it: along its rows
// (K-major) where K is its column index, down its columns (MN-major) where K is its row index, so
// nothing is transposed and the features and weights are read in place.  (Staging each operand of
// each contraction by itself, six segments wide and transposed where K was the row index, was 42
// launches and 0.47 of 1.60 ms at 4 samples of 2880 tokens; the step went from 1424 to 922 us.)
// The images' logits and their gradients are one batched contraction each.  The softmax, KL, RoPE and
// GELU steps and their derivatives are fp32, with fixed-order (deterministic) reductions.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cuda_bf16.h>

#include "kernels.h"
#include "ptx.cuh"

namespace mapk {
namespace {

// hi = bf16(x), mid = bf16(x - hi), lo = bf16(x - hi - mid): x = hi + mid + lo to about 24
// significant bits (both differences are exact in fp32).
struct Split3 { uint16_t h, m, l; };
__device__ __forceinline__ Split3 split3(float x) {
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  const __nv_bfloat16 l = __float2bfloat16_rn(r1 - __bfloat162float(m));
  return {__bfloat16_as_ushort(h), __bfloat16_as_ushort(m), __bfloat16_as_ushort(l)};
}
// Four consecutive values to the three segments (seg columns apart) at dst (8-byte stores).
__device__ __forceinline__ void store_split4(uint16_t* dst, long long seg, const float (&x)[4]) {
  Split3 s[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) s[u] = split3(x[u]);
  *reinterpret_cast<ushort4*>(dst) = make_ushort4(s[0].h, s[1].h, s[2].h, s[3].h);
  *reinterpret_cast<ushort4*>(dst + seg) = make_ushort4(s[0].m, s[1].m, s[2].m, s[3].m);
  *reinterpret_cast<ushort4*>(dst + 2 * seg) = make_ushort4(s[0].l, s[1].l, s[2].l, s[3].l);
}
__device__ __forceinline__ void store_split2(uint16_t* dst, long long seg, float x, float y) {
  const Split3 a = split3(x), b = split3(y);
  *reinterpret_cast<ushort2*>(dst) = make_ushort2(a.h, b.h);
  *reinterpret_cast<ushort2*>(dst + seg) = make_ushort2(a.m, b.m);
  *reinterpret_cast<ushort2*>(dst + 2 * seg) = make_ushort2(a.l, b.l);
}

// Four / two consecutive elements of a contraction's result, its K slices added in order.
__device__ __forceinline__ float4 load_result4(const TcResult& in, long long r, int c) {
  const float* p = in.p + r * in.ld + c;
  float4 x = *reinterpret_cast<const float4*>(p);
  for (int k = 1; k < in.ks; ++k) {
    const float4 y = *reinterpret_cast<const float4*>(p + k * in.stride);
    x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
  }
  return x;
}
__device__ __forceinline__ float2 load_result2(const TcResult& in, long long r, int c) {
  const float* p = in.p + r * in.ld + c;
  float2 x = *reinterpret_cast<const float2*>(p);
  for (int k = 1; k < in.ks; ++k) {
    const float2 y = *reinterpret_cast<const float2*>(p + k * in.stride);
    x.x += y.x; x.y += y.y;
  }
  return x;
}

// x Phi(x) and its derivative Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_and_grad(float x, float& grad) {
  const float Phi = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
  const float phi = 0.39894228040143268f * expf(-0.5f * x * x);
  grad = Phi + x * phi;
  return x * Phi;
}

// Elementwise steps and the staging of their result in one pass: a warp reads 128 columns of a row
// (16 bytes a lane) and writes them to the three segments of the staged matrix [rows, 3 cols].
// A block takes 128 columns of kColRows rows.
constexpr int kColRows = 64;                        // rows of a block, and of a partial column sum
constexpr int kActWarps = 8;

// x = GELU(in + bias), its derivative kept in fp32 for the backward pass (GELU; the error function is
// evaluated once for both), or x = in + bias.
template <bool GELU>
__global__ void __launch_bounds__(32 * kActWarps) act_split_kernel(TcResult in, const __nv_bfloat16* __restrict__ bias,
                                                                   long long rows, int cols, float* __restrict__ grad,
                                                                   uint16_t* __restrict__ dst) {
  pdl_enter();
  const int c = blockIdx.x * 128 + 4 * (threadIdx.x & 31), w = threadIdx.x >> 5;
  float b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) b[u] = __bfloat162float(bias[c + u]);
  const long long r0 = static_cast<long long>(blockIdx.y) * kColRows;
#pragma unroll 4
  for (int i = w; i < kColRows; i += kActWarps) {
    const long long r = r0 + i;
    if (r >= rows) break;
    const float4 v = load_result4(in, r, c);
    float x[4] = {v.x + b[0], v.y + b[1], v.z + b[2], v.w + b[3]};
    if (GELU) {
      float g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = gelu_and_grad(x[u], g[u]);
      *reinterpret_cast<float4*>(grad + r * cols + c) = make_float4(g[0], g[1], g[2], g[3]);
    }
    store_split4(dst + r * 3 * cols + c, cols, x);
  }
}

// x = in * grad (BACK) or in; part[block row][c] = the block's column sums of x.
template <bool BACK>
__global__ void __launch_bounds__(32 * kActWarps) back_split_kernel(TcResult in, const float* __restrict__ grad,
                                                                    long long rows, int cols,
                                                                    uint16_t* __restrict__ dst,
                                                                    float* __restrict__ part) {
  __shared__ float4 red[kActWarps][32];
  pdl_enter();
  const int lane = threadIdx.x & 31, c = blockIdx.x * 128 + 4 * lane, w = threadIdx.x >> 5;
  const long long r0 = static_cast<long long>(blockIdx.y) * kColRows;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int i = w; i < kColRows; i += kActWarps) {
    const long long r = r0 + i;
    if (r >= rows) break;
    const float4 v = load_result4(in, r, c);
    float x[4] = {v.x, v.y, v.z, v.w};
    if (BACK) {
      const float4 g = *reinterpret_cast<const float4*>(grad + r * cols + c);
      x[0] *= g.x;
      x[1] *= g.y;
      x[2] *= g.z;
      x[3] *= g.w;
    }
    s.x += x[0]; s.y += x[1]; s.z += x[2]; s.w += x[3];
    store_split4(dst + r * 3 * cols + c, cols, x);
  }
  red[w][lane] = s;
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int i = 1; i < kActWarps; ++i) {
      const float4 y = red[i][lane];
      s.x += y.x; s.y += y.y; s.z += y.z; s.w += y.w;
    }
    *reinterpret_cast<float4*>(part + static_cast<long long>(blockIdx.y) * cols + c) = s;
  }
}

// out[c] = sum over the nparts partial sums, in a fixed order (32 columns x 8 phases per block).
__global__ void __launch_bounds__(256) colsum_final_kernel(const float* __restrict__ part, int nparts, int cols,
                                                           float* __restrict__ out) {
  __shared__ float red[8][32];
  pdl_enter();
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, c = blockIdx.x * 32 + x;
  float s = 0.f;
  if (c < cols)
#pragma unroll 8
    for (int p = y; p < nparts; p += 8) s += part[static_cast<long long>(p) * cols + c];
  red[y][x] = s;
  __syncthreads();
  if (y == 0 && c < cols) {
    for (int i = 1; i < 8; ++i) s += red[i][x];
    out[c] = s;
  }
}

// RoPE on rows of width 2 * half (rotate-half pairs (i, i + half)): forward y = scale R(a) x, or
// backward y = scale R(-a) x, staged as three terms.  Row r sits at position pos[r] (pos !=
// nullptr) or r % pos_mod; the (cos, sin) table is [half][ld], position-minor.  Two pairs a thread.
template <bool BACKWARD>
__global__ void __launch_bounds__(256) rope_split_kernel(TcResult in, const int32_t* __restrict__ in_map,
                                                         long long rows, int half, const float2* __restrict__ tab,
                                                         int ld, const int32_t* __restrict__ pos, int pos_mod,
                                                         float scale, uint16_t* __restrict__ dst,
                                                         const int32_t* __restrict__ out_map) {
  pdl_enter();
  const int h2 = half / 2;
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long r = t / h2;
  if (r >= rows) return;
  const int i = 2 * static_cast<int>(t - r * h2);
  const int p = pos ? pos[r] : static_cast<int>(r % pos_mod);
  const long long ri = in_map ? in_map[r] : r, ro = out_map ? out_map[r] : r;
  const float2 ca = tab[static_cast<long long>(i) * ld + p], cb = tab[static_cast<long long>(i + 1) * ld + p];
  const float2 x1 = load_result2(in, ri, i), x2 = load_result2(in, ri, half + i);
  float2 y1, y2;
  if (BACKWARD) {
    y1 = make_float2(x1.x * ca.x + x2.x * ca.y, x1.y * cb.x + x2.y * cb.y);
    y2 = make_float2(x2.x * ca.x - x1.x * ca.y, x2.y * cb.x - x1.y * cb.y);
  } else {
    y1 = make_float2(x1.x * ca.x - x2.x * ca.y, x1.y * cb.x - x2.y * cb.y);
    y2 = make_float2(x2.x * ca.x + x1.x * ca.y, x2.y * cb.x + x1.y * cb.y);
  }
  const int d = 2 * half;
  uint16_t* o = dst + ro * 3 * d + i;
  store_split2(o, d, y1.x * scale, y1.y * scale);
  store_split2(o + half, d, y2.x * scale, y2.y * scale);
}

// One CTA per image: where its rows start in the padded question layout (the images before it, each
// rounded up to 64 rows), the padded row of each of its rows, and the image of each padded row.
__global__ void __launch_bounds__(256) distill_meta_kernel(const int32_t* __restrict__ len,
                                                           const int32_t* __restrict__ off, int B,
                                                           int32_t* __restrict__ poff, int32_t* __restrict__ prow,
                                                           int32_t* __restrict__ img) {
  __shared__ int32_t red[256];
  pdl_enter();
  const int b = blockIdx.x;
  int32_t s = 0;
  for (int i = threadIdx.x; i < b; i += 256) s += (len[i] + 63) & ~63;
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const int32_t base = red[0];
  const int n = len[b], np = (n + 63) & ~63;
  if (threadIdx.x == 0) poff[b] = base;
  for (int m = threadIdx.x; m < np; m += 256) {
    img[base + m] = m < n ? b : -1;
    if (m < n) prow[off[b] + m] = base + m;
  }
}

__global__ void __launch_bounds__(128) zero_pad_rows_kernel(uint4* __restrict__ x, int vec_per_row,
                                                            const int32_t* __restrict__ img) {
  pdl_enter();
  if (img[blockIdx.x] >= 0) return;
  uint4* row = x + static_cast<long long>(blockIdx.x) * vec_per_row;
  for (int v = threadIdx.x; v < vec_per_row; v += blockDim.x) row[v] = make_uint4(0u, 0u, 0u, 0u);
}

constexpr int kRowThreads = 256;

// Deterministic block sum (kRowThreads threads): warp trees, then warp 0 in order.
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = red[0];
    for (int w = 1; w < kRowThreads / 32; ++w) s += red[w];
    red[kRowThreads / 32] = s;
  }
  __syncthreads();
  const float r = red[kRowThreads / 32];
  __syncthreads();
  return r;
}
__device__ __forceinline__ float block_max(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = red[0];
    for (int w = 1; w < kRowThreads / 32; ++w) s = fmaxf(s, red[w]);
    red[kRowThreads / 32] = s;
  }
  __syncthreads();
  const float r = red[kRowThreads / 32];
  __syncthreads();
  return r;
}

// One CTA per padded question row: logits row -> softmax over the N visual tokens, in place.
__global__ void __launch_bounds__(kRowThreads) row_softmax_kernel(float* __restrict__ L, long long ld, int N,
                                                                  const int32_t* __restrict__ img) {
  __shared__ float red[kRowThreads / 32 + 1];
  pdl_enter();
  if (img[blockIdx.x] < 0) return;                  // padding row
  float* row = L + static_cast<long long>(blockIdx.x) * ld;
  float m = -INFINITY;
  for (int n = threadIdx.x; n < N; n += kRowThreads) m = fmaxf(m, row[n]);
  m = block_max(m, red);
  float s = 0.f;
  for (int n = threadIdx.x; n < N; n += kRowThreads) s += expf(row[n] - m);
  s = block_sum(s, red);
  const float inv = 1.0f / s;
  for (int n = threadIdx.x; n < N; n += kRowThreads) row[n] = expf(row[n] - m) * inv;
}

// Per image b (grid.y) and column block: p_hat[n] = mean_m s[m, n]; g[n] = -p*[n] / (B p_hat[n]);
// the block's share of D_KL(p* || p_hat) goes to part[b * nblk + blockIdx.x].  Eight rows' loads are
// in flight before their sums (in row order).
__global__ void __launch_bounds__(kRowThreads) phat_kl_kernel(const float* __restrict__ S, long long ld,
                                                              const int32_t* __restrict__ len,
                                                              const int32_t* __restrict__ poff,
                                                              const float* __restrict__ teacher, int N, int B,
                                                              float* __restrict__ p_hat, float* __restrict__ g,
                                                              float* __restrict__ part) {
  __shared__ float red[kRowThreads / 32 + 1];
  pdl_enter();
  const int b = blockIdx.y;
  const int n = blockIdx.x * kRowThreads + threadIdx.x;
  const int M = len[b];
  float kl = 0.f;
  if (n < N) {
    const float* col = S + static_cast<long long>(poff[b]) * ld + n;
    float acc = 0.f;
    int m = 0;
    for (; m + 8 <= M; m += 8) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = col[static_cast<long long>(m + u) * ld];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc += x[u];
    }
    for (; m < M; ++m) acc += col[static_cast<long long>(m) * ld];
    const float ph = acc / static_cast<float>(M);
    const float ps = teacher[static_cast<long long>(b) * N + n];
    p_hat[static_cast<long long>(b) * N + n] = ph;
    g[static_cast<long long>(b) * N + n] = -ps / (static_cast<float>(B) * ph);
    if (ps > 0.f) kl = ps * logf(ps / ph);
  }
  kl = block_sum(kl, red);
  if (threadIdx.x == 0) part[static_cast<long long>(b) * gridDim.x + blockIdx.x] = kl;
}

// loss = (1/B) sum over images and blocks of the partial divergences, in order.
__global__ void loss_reduce_kernel(const float* __restrict__ part, int n, int B, float* __restrict__ loss) {
  pdl_enter();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < n; ++i) s += part[i];
    *loss = s / static_cast<float>(B);
  }
}

// One CTA per padded question row m of image b: softmax backward of the mean,
//   dl[m, n] = s[m, n] (g[n] - sum_n' s[m, n'] g[n']) / M_b,
// staged as three terms (zeros in padding rows and columns).
__global__ void __launch_bounds__(kRowThreads) softmax_back_kernel(const float* __restrict__ S, long long ld,
                                                                   const int32_t* __restrict__ len,
                                                                   const int32_t* __restrict__ img,
                                                                   const float* __restrict__ g, int N,
                                                                   uint16_t* __restrict__ dst, int seg) {
  __shared__ float red[kRowThreads / 32 + 1];
  pdl_enter();
  const long long m = blockIdx.x;
  const int b = img[m];
  uint16_t* out = dst + m * 3 * seg;
  if (b < 0) {
    for (int n = 2 * threadIdx.x; n < 3 * seg; n += 2 * kRowThreads) *reinterpret_cast<uint32_t*>(out + n) = 0u;
    return;
  }
  const float inv_m = 1.0f / static_cast<float>(len[b]);
  const float* row = S + m * ld;
  const float* gb = g + static_cast<long long>(b) * N;
  float c = 0.f;
  for (int n = threadIdx.x; n < N; n += kRowThreads) c += row[n] * gb[n];
  c = block_sum(c, red);
  for (int n = 2 * threadIdx.x; n < seg; n += 2 * kRowThreads) {
    const float x = n < N ? row[n] * (gb[n] - c) * inv_m : 0.f;
    const float y = n + 1 < N ? row[n + 1] * (gb[n + 1] - c) * inv_m : 0.f;
    store_split2(out + n, seg, x, y);
  }
}

// C[i, j] = sum over the ks K slices of part[s * stride + i * ldp + j], in slice order.
__global__ void sum_slices_kernel(const float* __restrict__ part, int ks, long long stride, int M, int N,
                                  long long ldp, float* __restrict__ C, long long ldc) {
  pdl_enter();
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= static_cast<long long>(M) * N) return;
  const long long i = t / N, j = t - i * N;
  const float* p = part + i * ldp + j;
  float s = 0.f;
  for (int k = 0; k < ks; ++k) s += p[k * stride];
  C[i * ldc + j] = s;
}

}  // namespace

// Products of terms kept for each kind of operand pair (x = hi + mid + lo for an fp32 operand,
// exact for a bf16 one): everything down to about 2^-24 relative, so the result is as good as an
// fp32 product accumulated in fp32.
//   bf16 . bf16 : a.b                                           1 product
//   fp32 . bf16 : lo.b + mid.b + hi.b                           3 products
//   fp32 . fp32 : mm + hl + lh + hm + mh + hh                   6 products (ml, lm, ll are below 2^-24)
// One GEMM runs over the products' K side by side, smallest terms first, so that the tensor cores'
// fp32 accumulator adds the small terms while it is still small and runs only the last K / 16 steps
// at full magnitude (their additions are where the accumulation error comes from).
int tc_products(bool a_split, bool b_split) { return a_split && b_split ? 6 : (a_split || b_split ? 3 : 1); }

// K slices for a GEMM whose output has too few tiles to fill the GPU (the weight gradients over
// the token index, the per-image query gradients): enough slices to give every SM (or 2-SM
// pair) a unit, each slice at least 16 K blocks deep.  Mirrors launch_gemm's choice of the
// 1-SM tile for an output of at most 128 x 128 and of 2-SM 256 x 256 tiles otherwise.
int tc_ksplit(int M, int N, int K, int products, int num_sms) {
  const bool pair = !(M <= 128 && N <= 128);
  const int units = pair ? ((M + 127) / 128 + 1) / 2 * ((N + 255) / 256) : ((M + 127) / 128) * ((N + 127) / 128);
  const int slots = pair ? num_sms / 2 : num_sms;
  const int kbs = products * ((K + 63) / 64);
  if (units <= 0 || units * 2 > slots) return 1;
  int ks = std::min(slots / units, kbs / 16);
  return ks < 1 ? 1 : ks;
}

cudaError_t launch_tc_matmul(int M, int N, int K, const TcOperand& A, const TcOperand& B, const TcBatch& batch,
                             int ksplit, bool add, float* C, long long ldc, float* wsC, int num_sms, int* status,
                             long long wait_ns, cudaStream_t st, long long* launches, TcResult* res) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaErrorInvalidValue;
  GemmDesc d{};
  GemmProducts& q = d.pr;
  q.n = tc_products(A.seg > 0, B.seg > 0);
  q.kblocks = (K + 63) / 64;
  // terms 0 hi, 1 mid, 2 lo
  static const int kA6[6] = {1, 0, 2, 0, 1, 0}, kB6[6] = {1, 2, 0, 1, 0, 0}, kT3[3] = {2, 1, 0};
  for (int i = 0; i < q.n; ++i) {
    const int ta = q.n == 6 ? kA6[i] : (q.n == 3 ? kT3[i] : 0), tb = q.n == 6 ? kB6[i] : (q.n == 3 ? kT3[i] : 0);
    q.a_seg[i] = A.seg > 0 ? ta * A.seg : 0;
    q.b_seg[i] = B.seg > 0 ? tb * B.seg : 0;
  }
  q.a_mn = A.mn; q.b_mn = B.mn; q.a_cols = A.cols; q.b_cols = B.cols;
  q.a_off = batch.a_off; q.b_off = batch.b_off; q.k_count = batch.k_count;
  d.A = A.p; d.a_rows_total = A.rows; d.a_row_stride = batch.a_rows;
  d.B = B.p; d.b_rows_total = B.rows; d.b_row_stride = batch.b_rows;
  d.M = M; d.N = N; d.K = q.n * q.kblocks * 64; d.batch = batch.n;
  d.m_limit = batch.m_count;
  d.epi = EPI_F32; d.status = status; d.wait_ns = wait_ns;
  const long long crows = batch.n > 1 || batch.a_off ? batch.c_rows : M;
  if (launches) ++*launches;
  cudaError_t e;
  if (ksplit <= 1) {
    d.C = C; d.ldc = ldc; d.c_batch_stride = batch.c_stride;
    if (res) *res = TcResult{C, 1, 0, ldc};
    return launch_gemm(d, num_sms, st);
  }
  // K slices into wsC
  const long long ldp = (N + 3) / 4 * 4;
  d.C = wsC; d.ldc = ldp; d.c_batch_stride = batch.c_stride;
  d.ksplit = ksplit; d.c_split_stride = crows * ldp;
  if ((e = launch_gemm(d, num_sms, st)) != cudaSuccess) return e;
  if (res) *res = TcResult{wsC, ksplit, d.c_split_stride, ldp};
  if (!add) return cudaSuccess;
  const long long total = crows * N;
  if (launches) ++*launches;
  return launch_k(sum_slices_kernel, dim3(static_cast<unsigned>((total + 255) / 256)), dim3(256), 0, st,
                  static_cast<const float*>(wsC), ksplit, d.c_split_stride, static_cast<int>(crows), N, ldp, C, ldc);
}

cudaError_t launch_distill_meta(const int32_t* len, const int32_t* off, int B, int32_t* poff, int32_t* prow,
                                int32_t* img, cudaStream_t st) {
  return launch_k(distill_meta_kernel, dim3(B), dim3(256), 0, st, len, off, B, poff, prow, img);
}

namespace {
dim3 act_grid(long long rows, int cols) {
  return dim3(cols / 128, static_cast<unsigned>((rows + kColRows - 1) / kColRows));
}
}  // namespace

cudaError_t launch_act_split(bool gelu, const TcResult& in, const void* bias, long long rows, int cols, float* grad,
                             void* dst, cudaStream_t st) {
  if (cols % 128 != 0) return cudaErrorInvalidValue;
  const __nv_bfloat16* b = static_cast<const __nv_bfloat16*>(bias);
  uint16_t* d = static_cast<uint16_t*>(dst);
  if (gelu) return launch_k(act_split_kernel<true>, act_grid(rows, cols), dim3(32 * kActWarps), 0, st, in, b, rows, cols, grad, d);
  return launch_k(act_split_kernel<false>, act_grid(rows, cols), dim3(32 * kActWarps), 0, st, in, b, rows, cols, grad, d);
}

cudaError_t launch_back_split(const TcResult& in, const float* grad, long long rows, int cols, void* dst, float* part,
                              float* colsum, cudaStream_t st) {
  if (cols % 128 != 0) return cudaErrorInvalidValue;
  uint16_t* d = static_cast<uint16_t*>(dst);
  const dim3 grid = act_grid(rows, cols);
  const cudaError_t e =
      grad ? launch_k(back_split_kernel<true>, grid, dim3(32 * kActWarps), 0, st, in, grad, rows, cols, d, part)
           : launch_k(back_split_kernel<false>, grid, dim3(32 * kActWarps), 0, st, in, grad, rows, cols, d, part);
  if (e != cudaSuccess) return e;
  return launch_k(colsum_final_kernel, dim3((cols + 31) / 32), dim3(256), 0, st, static_cast<const float*>(part),
                  static_cast<int>(grid.y), cols, colsum);
}

cudaError_t launch_rope_split(bool backward, const TcResult& in, const int32_t* in_map, long long rows, int d,
                              const float2* tab, int ld, const int32_t* pos, int pos_mod, float scale, void* dst,
                              const int32_t* out_map, cudaStream_t st) {
  const long long total = rows * (d / 4);
  const dim3 grid(static_cast<unsigned>((total + 255) / 256));
  uint16_t* o = static_cast<uint16_t*>(dst);
  if (backward)
    return launch_k(rope_split_kernel<true>, grid, dim3(256), 0, st, in, in_map, rows, d / 2, tab, ld, pos, pos_mod,
                    scale, o, out_map);
  return launch_k(rope_split_kernel<false>, grid, dim3(256), 0, st, in, in_map, rows, d / 2, tab, ld, pos, pos_mod,
                  scale, o, out_map);
}

cudaError_t launch_distill_loss_grad(float* S, long long ld, long long prows, const int32_t* len,
                                     const int32_t* poff, const int32_t* img, const float* teacher, int B, int N,
                                     float* p_hat, float* g, float* part, float* loss, void* dst, int seg,
                                     cudaStream_t st) {
  const dim3 rows(static_cast<unsigned>(prows));
  cudaError_t e = launch_k(row_softmax_kernel, rows, dim3(kRowThreads), 0, st, S, ld, N, img);
  if (e != cudaSuccess) return e;
  const int nblk = (N + kRowThreads - 1) / kRowThreads;
  e = launch_k(phat_kl_kernel, dim3(nblk, B), dim3(kRowThreads), 0, st, static_cast<const float*>(S), ld, len, poff,
               teacher, N, B, p_hat, g, part);
  if (e != cudaSuccess) return e;
  e = launch_k(loss_reduce_kernel, dim3(1), dim3(32), 0, st, static_cast<const float*>(part), nblk * B, B, loss);
  if (e != cudaSuccess) return e;
  return launch_k(softmax_back_kernel, rows, dim3(kRowThreads), 0, st, static_cast<const float*>(S), ld, len, img,
                  static_cast<const float*>(g), N, static_cast<uint16_t*>(dst), seg);
}

cudaError_t launch_zero_pad_rows(void* x, int cols, const int32_t* img, long long prows, cudaStream_t st) {
  if (cols % 8 != 0) return cudaErrorInvalidValue;
  return launch_k(zero_pad_rows_kernel, dim3(static_cast<unsigned>(prows)), dim3(128), 0, st, static_cast<uint4*>(x),
                  cols / 8, img);
}

}  // namespace mapk
