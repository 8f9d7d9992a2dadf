// Host-side launchers of the CUDA kernels (internal to libmap_gb300).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mapk {

// Products of two tokens' features (selection) are fp32 sums of this many K slices, slice s the 64-column
// blocks s KB / kGramSlices ..., added in slice order: in the Gram kernel, where a CTA of the cluster takes a slice,
// and in EPI_PROJECT alike.  What is subtracted from or divided by each other (a Gram entry and the norms
// it meets) must be the same sum: the tensor cores lose up to an ulp a 16-term step, and with two orders exact
// copies of R0 tokens counted as independent (r^2 > tau ||v||^2) from 4096 columns on.
constexpr int kGramSlices = 8;

// *_SPLIT epilogues store an fp32 activation x as two bf16 halves, hi = bf16(x) at
// column c and lo = bf16(x - hi) at column N + c of a [rows, 2N] buffer, so that the next
// layer can consume ~16 significant bits through a bf16 GEMM: [hi | lo] @ [W | W]^T.
// EPI_ROPE_SPLIT3 applies RoPE (and `scale`) and stores the vector as three bf16
// segments, [hi | lo | hi] (split_kind 0, keys) or [hi | hi | lo] (split_kind 1, queries),
// so that one bf16 GEMM with K = 3 dp gives q.k to about 16 significant bits; it can also
// store the fp32 vector to `aux`.
// EPI_SM_STATS / EPI_SM_MEAN are the two passes of Eq. 3 over a logits tile (rows =
// visual tokens, columns = question tokens): per-column max / sum of exp over each
// 32-row slab, then per-row mean over columns of exp(l - max) / sum.
// EPI_PROJECT: rows = visual tokens, columns = the R0 basis tokens' rows (Gram entries
// <v_n, v_r>, sums of K slices); the epilogue solves for the tokens' Cholesky coordinates against the R0
// basis (L staged in shared memory); ||v_n||^2 is the diagonal of an A A^T product that the
// MMA thread accumulates from the same shared-memory tiles.  It writes the exact residual,
// value and coordinate cache of every candidate token (see select.cu).
enum Epi { EPI_GELU_BF16 = 0, EPI_BIAS_BF16 = 1, EPI_ROPE_F32 = 2, EPI_F32 = 3, EPI_GELU_SPLIT = 4,
           EPI_BIAS_SPLIT = 5, EPI_ROPE_SPLIT3 = 6, EPI_SM_STATS = 7, EPI_SM_MEAN = 8, EPI_PROJECT = 9 };

// Inputs and outputs of the EPI_PROJECT epilogue (device pointers).
struct ProjArgs {
  const uint8_t* state;        // [B, N] 0 = candidate
  const float* scores;         // [B, N] p_hat
  float* Ec; int KP;           // coordinate cache rows [B, N, KP]
  const int32_t* basis_tok;    // [B, Kcap]
  const float* rnorm;          // [B, Kcap]
  const int32_t* nbasis;       // [B] basis size after R0 (<= 128)
  int Kcap;
  float lambda, tau;
  float* r2; float* U; float* sqn; int32_t* cstep;   // [B, N] outputs
};

// EPI_F32 as a sum of products of column segments: C = sum_p A_p B_p^T, where A_p (B_p) is the
// operand's array from column a_seg[p] (b_seg[p]) on.  An array of a_cols columns (row stride too)
// is K-major (its rows are the operand's rows, K runs along a row) or, with a_mn, MN-major (its
// rows are the K index, the operand's rows run along a row): no operand is transposed in memory.
// Batched: an operand's array rows of entry b start at a_off[b] (device) or b * a_row_stride,
// likewise B's; K per entry is k_count[b] (device; rows past it up to the next multiple of 64 must
// be zero in one operand) or 64 * kblocks.  With a_off and a K-major A, C has A's rows.
constexpr int kMaxProducts = 6;
struct GemmProducts {
  int n;                       // 0: a plain product
  int kblocks;                 // 64-wide K blocks of one product (the most over the batch)
  int a_seg[kMaxProducts], b_seg[kMaxProducts];
  int a_mn, b_mn, a_cols, b_cols;
  const int* a_off; const int* b_off; const int* k_count;
};

// Batched C = epi(A @ B^T): A rows [batch][a_row_stride] x K, B rows [batch][b_row_stride] x K
// (both bf16, K contiguous, tightly packed 2D arrays of a_rows_total / b_rows_total rows).
struct GemmDesc {
  const void* A; long long a_rows_total; int a_row_stride;
  const void* B; long long b_rows_total; int b_row_stride;
  int M, N, K, batch;
  const int* n_limit;                   // per-batch output-column limit (device) or nullptr
  void* C; long long ldc; long long c_batch_stride;   // elements
  const void* bias;                     // bf16 [N] or nullptr
  const float2* rope; int rope_half;    // (cos, sin) table [rope_half][rope_ld]: position-minor, so
  int rope_ld = 0;                      // lanes (consecutive rows) read consecutive entries
  const int* pos; int pos_mod;          // per-row positions (device) or row % pos_mod
  int epi;
  int* status;
  // EPI_ROPE_SPLIT3
  int split_kind = 0; float scale = 1.f; float* aux = nullptr;
  // batched B rows at per-batch offsets (device) instead of b * b_row_stride
  const int* b_off = nullptr;
  // EPI_SM_STATS: partial (max, sum) per 32-row slab [batch][m_tiles * 4][stat_ld] (float2)
  // EPI_SM_MEAN:  final (max + ln sum, 1/sum) per column [batch][stat_ld]; output C = scores
  //               [batch][M] when one column tile covers all columns; with stat_parts > 0, stats is the
  //               partial array of that many slabs instead, combined by every tile for its columns
  float2* stats = nullptr; int stat_ld = 0; int stat_parts = 0;
  const int* col_count = nullptr;       // per-batch number of valid columns (M_b)
  // B rows at b * b_row_stride + b_base
  int b_base = 0;
  ProjArgs proj{};
  // A has a_kwrap columns; its K coordinate wraps (k mod a_kwrap), so a K-segment of A can
  // be read twice against different B segments (0: A has K columns)
  int a_kwrap = 0;
  // split3 = 1 (with K = 3 Dh, A = [hi | lo] and B = [W_hi | W_hi | W_lo]): K blocks are taken
  // as (hi_j, W_hi_j), (hi_j, W_lo_j) for every j, then (lo_j, W_hi_j), so each block of A_hi
  // is read twice back to back (the second time from L2)
  int split3 = 0;
  const float* biasf = nullptr;         // EPI_ROPE_SPLIT3: fp32 bias [N] added before RoPE
  // Batch entries to process (device): blist[0 .. *bcount) instead of 0 .. batch-1, so that a
  // launch over a few active images spreads their tiles over all SMs (grid sized for batch)
  const int* blist = nullptr; const int* bcount = nullptr;
  // Per-batch number of valid A rows (device) or nullptr: rows at or past it are treated as
  // absent (EPI_SM_STATS: excluded from the column statistics; EPI_SM_MEAN: output 0)
  const int* m_limit = nullptr;
  // Limit (ns) of the producer / MMA / epilogue waits; 0 = the default 2 s.  The waits that
  // let in-flight copies and MMAs land before an aborting CTA exits keep the default.
  long long wait_ns = 0;
  // EPI_F32 split-K: ksplit K slices, each unit one slice of a tile, slice s writing its partial
  // sum at C + s * c_split_stride (elements, a multiple of 4); the caller adds the slices
  int ksplit = 1; long long c_split_stride = 0;
  GemmProducts pr{};
  // EPI_GELU_SPLIT, N % 256 == 0: columns of a tile, 64, 128, 192 or 256 (0)
  int tile_n = 0;
  // EPI_GELU_SPLIT, EPI_ROPE_SPLIT3: the rows are segments of seg_len rows, of which the first
  // seg_valid[s] (device) hold data; tiles without such rows are skipped (nullptr: all rows)
  const int* seg_valid = nullptr; int seg_len = 0;
};

// EPI_F32 results that box stores can write: every batch entry's (or K slice's) rows and columns end at
// M and N, at a fixed distance from the next one's.  N % 64 == 0: a warp's two staging buffers take the
// 32-column chunks of a tile in turn, from the first one in every tile, and a chunk waits for all stores but the
// last; after a tile of an odd number of chunks that last one might still read the buffer.
inline bool f32_box_store(const GemmDesc& d) {
  return d.epi == EPI_F32 && d.N % 64 == 0 && (d.batch == 1 || d.ksplit == 1) && !d.n_limit && !d.m_limit &&
         !d.blist && (!d.pr.a_off || d.pr.a_mn);
}

// tile_n of the first layer of both branches (m_vis and m_text rows, N columns).
int predictor_tile_width(long long m_vis, long long m_text, int N, int K, int num_sms);
// Returns cudaSuccess, or an error for an unsupported shape (cudaErrorInvalidValue).
cudaError_t launch_gemm(const GemmDesc& d, int num_sms, cudaStream_t st);
// Both in one launch: two row groups that share N, K, the epilogue and its table (EPI_GELU_SPLIT,
// EPI_ROPE_SPLIT3).
cudaError_t launch_gemm_groups(const GemmDesc& d, const GemmDesc& d2, int num_sms, cudaStream_t st);

// Folds a projection after a linear layer into one matrix: W = Wp W2 ([dp, Dh] = [dp, Dh] x
// [Dh, Dh]) and bias = Wp b2, accumulated in fp64 from the bf16 inputs.  W is stored as the
// bf16 rows [hi | hi | lo] ([dp, 3 Dh], hi = bf16(W), lo = bf16(W - hi)) for activations laid
// out [hi | lo] and read with the K-wrap [hi | lo | hi]; bias in fp32.
cudaError_t launch_fold_weights(const void* Wp, const void* W2, const void* b2, int dp, int Dh, void* out,
                                float* bias_out, cudaStream_t st);

// Per-image question metadata written on the device from values passed as kernel parameters
// (no host-to-device copy, so nothing queues behind bulk input copies on the copy engines):
// off[b] = first query row of image b (off[B] = total), len[b], pos[row] = N + m for the
// m-th question token of its image.  lens has B entries; offs are their exclusive prefix sums.
// With nv (host, B entries: valid visual tokens per image) the positions are nv[b] + m and
// nvalid[b] = nv[b] is written too (nvalid may be nullptr).
cudaError_t launch_query_meta(const int32_t* lens, const long long* offs, int B, int N, int32_t* off, int32_t* len,
                              int32_t* pos, const int32_t* nv, int32_t* nvalid, cudaStream_t st);
// dst[0 .. n) = host[0 .. n), passed as kernel parameters (no copy engine).
cudaError_t launch_put_ints(const int32_t* host, int n, int32_t* dst, cudaStream_t st);
// Copies two device ints into host-mapped memory (device aliases of pinned host words).
cudaError_t launch_flags_to_host(const int32_t* a, const int* b, int32_t* a_host_dev, int* b_host_dev, cudaStream_t st);

// Squared row norms of bf16 rows: out[r] = sum_d x[r, d]^2 (fp32).
cudaError_t launch_row_sqnorm(const void* x, long long rows, int D, float* out, cudaStream_t st);

// scores[b, n] = sum_t part[b, t, n] over the column tiles (of `cols` question tokens, n_tiles slots an
// image) that hold image b's lens[b] tokens; the other slots are never written.
cudaError_t launch_sum_tiles(const float* part, int B, int N, int n_tiles, int cols, const int* lens, float* scores,
                             cudaStream_t st);

// Combines the per-slab softmax statistics into (max + ln sum, 1/sum) per question token:
// part [B][nparts][ld] -> fin [B][ld], columns < lens[b].
cudaError_t launch_stats_combine(const float2* part, int B, int nparts, int ld, const int* lens, float2* fin,
                                 cudaStream_t st);

// Gather rows: out[b, j, :] = V[b, idx[b, j], :].
cudaError_t launch_gather(const void* V, const int32_t* idx, int B, int N, int k, int D, void* out,
                          int* status, cudaStream_t st);

// Hand-off sequence per image: the kept rows V[b, idx[b, j]] (j < k), then the image's
// lens[b] question rows of T (packed in image order); pos = the kept index or n_b + m, plus
// pos_offset, with n_b = nv[b] (host; nullptr: N).  Indices outside [0, n_b) are not copied:
// pos = -1 and ST_BADINDEX in *status.
cudaError_t launch_assemble(const void* V, const int32_t* idx, const void* T, const int32_t* lens, const int32_t* nv,
                            int B, int N, int k, int D, int pos_offset, void* seq, int32_t* pos, int* status,
                            cudaStream_t st);

// ------------------------------------------------------------------ distillation step (fp32)
// A bf16 operand of a contraction: element (i, k) = p[i * cols + k] (mn = 0) or p[k * cols + i]
// (mn = 1), `rows` array rows.  seg > 0: an fp32 operand as three bf16 terms hi, mid, lo at columns
// 0, seg and 2 seg (split-bf16 products to fp32 accuracy, see distill.cu); 0: exact bf16.
struct TcOperand {
  const void* p; long long rows; int cols; int seg; int mn;
};
// Result of a contraction before its K slices are added: sum over s < ks of p[s * stride + row * ld
// + col] (ks = 1: the result itself).
struct TcResult {
  const float* p; int ks; long long stride; long long ld;
};
// Batch of a contraction (device arrays; batch 1: none), as in GemmProducts / GemmDesc.
struct TcBatch {
  int n = 1;
  const int* a_off = nullptr; int a_rows = 0;        // array rows of A per entry
  const int* b_off = nullptr; int b_rows = 0;
  const int* m_count = nullptr;                      // rows of C per entry
  const int* k_count = nullptr;
  long long c_stride = 0;                            // C elements per entry (without a_off)
  long long c_rows = 0;                              // rows of C over the whole batch
};
// K slices launch_tc_matmul takes for an M x N output over K.
int tc_ksplit(int M, int N, int K, int products, int num_sms);
int tc_products(bool a_split, bool b_split);
// C[i, j] = sum_k A(i, k) B(j, k) on the tcgen05 GEMM, fp32 out, deterministic (fixed order).  With
// one K slice the result is in C (16-byte aligned, ldc % 4 == 0); with more, the slices are in wsC
// and, with add = true, their sum in C (else the consumer adds them).
cudaError_t launch_tc_matmul(int M, int N, int K, const TcOperand& A, const TcOperand& B, const TcBatch& batch,
                             int ksplit, bool add, float* C, long long ldc, float* wsC, int num_sms, int* status,
                             long long wait_ns, cudaStream_t st, long long* launches, TcResult* res);
// Rows of the padded question layout (each image's rows start at a multiple of 64): poff[b], the
// padded row of every question row, and the image of every padded row (-1: padding).
cudaError_t launch_distill_meta(const int32_t* len, const int32_t* off, int B, int32_t* poff, int32_t* prow,
                                int32_t* img, cudaStream_t st);
// x = GELU(in + bias) (gelu: GELU'(in + bias) goes to grad) or in + bias, as three bf16 terms [rows, 3 cols].
cudaError_t launch_act_split(bool gelu, const TcResult& in, const void* bias, long long rows, int cols, float* grad,
                             void* dst, cudaStream_t st);
// x = in * grad (if given) or in, as three bf16 terms, and its column sums (part: kColRows-row
// partial sums, ceil(rows / 64) * cols floats).
cudaError_t launch_back_split(const TcResult& in, const float* grad, long long rows, int cols, void* dst, float* part,
                              float* colsum, cudaStream_t st);
// RoPE (or its transpose) of in [rows, d] times scale, as three bf16 terms at row in_map / out_map
// (nullptr: the row itself).  Position pos[r] or r % pos_mod.
cudaError_t launch_rope_split(bool backward, const TcResult& in, const int32_t* in_map, long long rows, int d,
                              const float2* tab, int ld, const int32_t* pos, int pos_mod, float scale, void* dst,
                              const int32_t* out_map, cudaStream_t st);
// S [padded rows, ld] logits -> p_hat [B, N], g = dL/dp_hat, *loss = mean_b D_KL(teacher_b ||
// p_hat_b), and dL/dlogits as three bf16 terms [padded rows, 3 seg] (zero in padding rows and past
// column N).  part: B * ceil(N / 256) floats.  S is overwritten.
cudaError_t launch_distill_loss_grad(float* S, long long ld, long long prows, const int32_t* len,
                                     const int32_t* poff, const int32_t* img, const float* teacher, int B, int N,
                                     float* p_hat, float* g, float* part, float* loss, void* dst, int seg,
                                     cudaStream_t st);
// Zeroes the padding rows of a [padded rows, cols] bf16 array.
cudaError_t launch_zero_pad_rows(void* x, int cols, const int32_t* img, long long prows, cudaStream_t st);

}  // namespace mapk
