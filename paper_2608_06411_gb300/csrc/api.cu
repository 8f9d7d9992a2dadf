// C ABI of libmap_gb300 (include/map_gb300.h): context, workspace, argument checks and
// the orchestration of the kernels for score (Eq. 3), select (Eq. 4) and gather.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/map_gb300.h"
#include "kernels.h"
#include "ptx.cuh"
#include "select.h"

using mapk::GemmDesc;

namespace {

constexpr int kMaxKDiverse = 768;   // k limit when the diversity term is on (the coordinate update
                                    // stages slot rows and 32 basis rows of k floats in shared memory)
constexpr int kProjMaxBasis = 128;  // basis vectors one projection pass takes
constexpr int kMaxK = 4096;
constexpr int kCombineInTile = 28;  // most softmax statistics a thread combines in Eq. 3's second pass itself
constexpr int kMaxN = 16384;

struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
};

struct TimedPair { cudaEvent_t a, b; int id; };

}  // namespace

struct map_ctx {
  map_config cfg{};
  int device = 0, num_sms = 148;
  void* w[10] = {};                 // wT1 bT1 wT2 bT2 wQ wV1 bV1 wV2 bV2 wK (device bf16)
  // W_Q f_T layer 2 and W_K f_V layer 2 folded (no nonlinearity between them): bf16 rows
  // [hi | hi | lo] of W_Q W_T2 / W_K W_V2 ([dp, 3 Dh]) and fp32 biases W_Q b_T2 / W_K b_V2
  void* wqt = nullptr; void* wkv = nullptr; float* bqt = nullptr; float* bkv = nullptr;
  DevBuf rope;  int rope_rows = 0;
  DevBuf h1, kb, th1, qb, stats, qoff, post, sqn, pmean, snv, dist;
  // selection
  DevBuf sU, sr2, scstep, sstate, sEc, spicks, sr0, sbt, srn, ssmall, stheta, saslot, sVg, sG;
  // map_prune staging
  DevBuf pvis, ptext, pout, pkeep, pscores;
  int* status = nullptr;            // device status word
  int* h_status = nullptr;          // pinned, mapped
  int32_t* h_done = nullptr;        // pinned, mapped
  int* h_status_dev = nullptr; int32_t* h_done_dev = nullptr;   // their device aliases
  cudaStream_t s_in = nullptr, s_out = nullptr;   // map_prune copy streams (host buffers)
  cudaStream_t s_aux = nullptr;     // question branch of the distillation step, beside the visual one
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  bool timing = false;
  std::vector<TimedPair> pairs;
  std::vector<cudaEvent_t> free_events;
  double t_ms[MAP_K_NUM] = {};
  long long t_n[MAP_K_NUM] = {};
  map_counters counters{};
  int deferred = MAP_OK;
  long long wait_ns = 0;            // GEMM role-wait limit (0: the kernels' default)
  mapk::SelLoopCache* loops = nullptr;   // cached graphs of the selection's device-side round loop
  long long* loop_iters_total = nullptr; // device: loop iterations run so far (one round each)
};

namespace {

int cuda_err(cudaError_t e) { return e == cudaSuccess ? MAP_OK : (e == cudaErrorMemoryAllocation ? MAP_ENOMEM : MAP_ECUDA); }

#define MAP_TRY(expr)                      \
  do {                                     \
    int _rc = (expr);                      \
    if (_rc != MAP_OK) return _rc;         \
  } while (0)
#define CU_TRY(expr) MAP_TRY(cuda_err(expr))

int ensure(DevBuf& b, size_t bytes) {
  if (bytes <= b.cap) return MAP_OK;
  if (b.p) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return MAP_ECUDA;
    cudaFree(b.p);
    b.p = nullptr;
    b.cap = 0;
  }
  size_t want = bytes + bytes / 8 + 256;
  if (cudaMalloc(&b.p, want) != cudaSuccess) {
    cudaGetLastError();
    return MAP_ENOMEM;
  }
  b.cap = want;
  return MAP_OK;
}

void release(DevBuf& b) {
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.cap = 0;
}

cudaEvent_t take_event(map_ctx* c) {
  if (!c->free_events.empty()) {
    cudaEvent_t e = c->free_events.back();
    c->free_events.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

// Brackets a launch with CUDA events when timing is on.
struct Timed {
  map_ctx* c; cudaStream_t st; int id; cudaEvent_t a = nullptr;
  Timed(map_ctx* c_, cudaStream_t st_, int id_) : c(c_), st(st_), id(id_) {
    if (c->timing) { a = take_event(c); cudaEventRecord(a, st); }
  }
  ~Timed() {
    if (a) {
      cudaEvent_t b = take_event(c);
      cudaEventRecord(b, st);
      c->pairs.push_back({a, b, id});
    }
  }
};

int dev_status_error(int st) {
  if (st & mapk::ST_TIMEOUT) return MAP_ETIMEOUT;
  if (st) return MAP_EINTERNAL;
  return MAP_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

int check_config(const map_config* c) {
  if (!c) return MAP_EINVAL;
  if (c->D <= 0 || c->D % 64 != 0) return MAP_EINVAL;
  if (c->Dh <= 0 || c->Dh % 256 != 0) return MAP_EINVAL;
  if (c->dp != 64 && c->dp != 128) return MAP_EINVAL;
  if (!(c->rope_theta > 0.f)) return MAP_EINVAL;
  if (!(c->lambda >= 0.f) || !(c->tau >= 0.f) || !(c->k0_frac >= 0.f)) return MAP_EINVAL;
  return MAP_OK;
}

int resolve_k0(const map_config& c, int K) {
  long long k0 = c.k0_abs >= 0 ? c.k0_abs : static_cast<long long>(std::floor(static_cast<double>(c.k0_frac) * K));
  if (k0 < 0) k0 = 0;
  if (k0 > K) k0 = K;
  return static_cast<int>(k0);
}

// RoPE table (cos, sin) of pos * theta^(-2i/dp), i < dp/2, for pos < rows; computed in
// double on the host, stored as float.
int ensure_rope(map_ctx* c, int rows_needed) {
  if (rows_needed <= c->rope_rows) return MAP_OK;
  const int rows = ((rows_needed + 1023) / 1024) * 1024;
  const int half = c->cfg.dp / 2;
  std::vector<float2> tab(static_cast<size_t>(rows) * half);
  for (int p = 0; p < rows; ++p)
    for (int i = 0; i < half; ++i) {
      const double f = std::pow(static_cast<double>(c->cfg.rope_theta), -2.0 * i / c->cfg.dp);
      const double a = p * f;
      tab[static_cast<size_t>(i) * rows + p] = make_float2(static_cast<float>(std::cos(a)), static_cast<float>(std::sin(a)));
    }
  MAP_TRY(ensure(c->rope, tab.size() * sizeof(float2)));
  CU_TRY(cudaMemcpy(c->rope.p, tab.data(), tab.size() * sizeof(float2), cudaMemcpyHostToDevice));
  c->rope_rows = rows;
  return MAP_OK;
}


int gemm(map_ctx* c, const GemmDesc& d, cudaStream_t st) {
  ++c->counters.launches;
  GemmDesc dd = d;
  dd.wait_ns = c->wait_ns;
  cudaError_t e = mapk::launch_gemm(dd, c->num_sms, st);
  if (e == cudaErrorInvalidValue) return MAP_EUNSUPPORTED;
  return cuda_err(e);
}

// The second stream of the question branch and its fork and join events.
int ensure_aux(map_ctx* c) {
  if (!c->s_aux) CU_TRY(cudaStreamCreateWithFlags(&c->s_aux, cudaStreamNonBlocking));
  if (!c->ev_fork) CU_TRY(cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming));
  if (!c->ev_join) CU_TRY(cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming));
  return MAP_OK;
}

GemmDesc linear_desc(map_ctx* c, const void* x, long long rows, int K, const void* w, int Nout, const void* bias,
                     void* y, int epi) {
  GemmDesc d{};
  d.A = x; d.a_rows_total = rows; d.a_row_stride = 0;
  d.B = w; d.b_rows_total = Nout; d.b_row_stride = 0;
  d.M = static_cast<int>(rows); d.N = Nout; d.K = K; d.batch = 1;
  d.n_limit = nullptr; d.C = y; d.ldc = Nout; d.c_batch_stride = 0;
  d.bias = bias; d.rope = nullptr; d.rope_half = c->cfg.dp / 2; d.pos = nullptr; d.pos_mod = 1;
  d.epi = epi; d.status = c->status;
  return d;
}

// Predictor of one modality (Eq. 3): x [rows, D] -> RoPE(Wp f(x)) * scale [rows, dp] with
// f = Linear -> GELU -> Linear, stored as three bf16 segments [rows, 3 dp] (split_kind 0:
// hi|lo|hi, 1: hi|hi|lo) and, if aux is given, as fp32 too.  The hidden activation
// h1 = GELU(W1 x + b1) is kept as a bf16 hi/lo pair [rows, 2 Dh] (about 16 significant bits);
// the second layer and the projection are one folded matrix Wf = Wp W2 with bias Wp b2.
struct Modality {
  const void* x; long long rows;
  const void* w1; const void* b1; const void* wf; const float* bf;
  void* h1; void* out3; int split_kind; float scale; float* aux;
  const int* pos; int pos_mod;
  const int* seg_valid; int seg_len;                 // rows that hold data (GemmDesc)
};

GemmDesc layer1_desc(map_ctx* c, const Modality& m, int tile_n) {
  const map_config& g = c->cfg;
  GemmDesc d = linear_desc(c, m.x, m.rows, g.D, m.w1, g.Dh, m.b1, m.h1, mapk::EPI_GELU_SPLIT);
  d.ldc = 2LL * g.Dh;
  d.tile_n = tile_n;
  d.seg_valid = m.seg_valid; d.seg_len = m.seg_len;
  return d;
}

GemmDesc projection_desc(map_ctx* c, const Modality& m) {
  const map_config& g = c->cfg;
  // K = 3 Dh: h_hi Wf_hi + h_hi Wf_lo + h_lo Wf_hi, A = [hi | lo] against
  // [Wf_hi | Wf_hi | Wf_lo], each block of h_hi used twice in a row (split3 K order)
  GemmDesc d = linear_desc(c, m.h1, m.rows, 3 * g.Dh, m.wf, g.dp, nullptr, m.out3, mapk::EPI_ROPE_SPLIT3);
  d.a_kwrap = 2 * g.Dh;
  d.split3 = 1;
  d.biasf = m.bf;
  d.ldc = 3LL * g.dp;
  d.rope = static_cast<const float2*>(c->rope.p);
  d.rope_ld = c->rope_rows;
  d.pos = g.rope_on ? m.pos : nullptr;      // without RoPE every position is 0: cos 1, sin 0
  d.pos_mod = g.rope_on ? m.pos_mod : 1;
  d.split_kind = m.split_kind;
  d.scale = m.scale;
  d.aux = m.aux;
  d.seg_valid = m.seg_valid; d.seg_len = m.seg_len;
  return d;
}

int gemm_groups(map_ctx* c, GemmDesc d, GemmDesc d2, cudaStream_t st) {
  ++c->counters.launches;
  d.wait_ns = d2.wait_ns = c->wait_ns;
  cudaError_t e = mapk::launch_gemm_groups(d, d2, c->num_sms, st);
  if (e == cudaErrorInvalidValue) return MAP_EUNSUPPORTED;
  return cuda_err(e);
}

// Both modalities, a layer of both in one launch: the question rows' tiles, too few for the chip,
// fill the visual rows' last wave instead of taking waves and a launch chain of their own (on a second
// stream they ran after the visual ones wherever those fill the chip: 95 of 2180 us with 64 images).
// With event timing on, each layer of each modality is its own launch.
int predictor(map_ctx* c, const Modality& vis, const Modality& text, int tile_n, cudaStream_t st) {
  if (!c->timing) {
    MAP_TRY(gemm_groups(c, layer1_desc(c, vis, tile_n), layer1_desc(c, text, tile_n), st));
    return gemm_groups(c, projection_desc(c, vis), projection_desc(c, text), st);
  }
  {
    Timed t(c, st, MAP_K_GEMM_TEXT);
    MAP_TRY(gemm(c, layer1_desc(c, text, tile_n), st));
    MAP_TRY(gemm(c, projection_desc(c, text), st));
  }
  {
    Timed t(c, st, MAP_K_GEMM_FV1);
    MAP_TRY(gemm(c, layer1_desc(c, vis, tile_n), st));
  }
  Timed t(c, st, MAP_K_GEMM_WK);
  return gemm(c, projection_desc(c, vis), st);
}

// nv (host, B entries, or nullptr = every image has N tokens): valid visual tokens per image;
// rows at or past nv[b] are padding, excluded from Eq. 3 (their score is 0).
int score_impl(map_ctx* c, const void* text, const void* vis, const int32_t* lens, const int32_t* nv, int B, int N,
               float* scores, float* q_out, float* k_out, cudaStream_t st) {
  if (!c || !text || !vis || !lens || !scores) return MAP_EINVAL;
  if (B < 1 || N < 1) return MAP_EINVAL;
  if (nv)
    for (int b = 0; b < B; ++b)
      if (nv[b] < 1 || nv[b] > N) return MAP_EINVAL;
  if (!aligned16(text) || !aligned16(vis)) return MAP_EINVAL;
  long long total_m = 0;
  int max_m = 0;
  for (int b = 0; b < B; ++b) {
    if (lens[b] < 1) return MAP_EINVAL;
    total_m += lens[b];
    max_m = lens[b] > max_m ? lens[b] : max_m;
  }
  if (total_m > (1ll << 30) || static_cast<long long>(B) * N > (1ll << 30)) return MAP_EUNSUPPORTED;
  const map_config& g = c->cfg;
  CU_TRY(cudaSetDevice(c->device));
  MAP_TRY(ensure_rope(c, g.rope_on ? N + max_m + 1 : 1));
  // per-image query offsets, lengths and question-token positions N + m, written on the device
  const size_t off_bytes = static_cast<size_t>(B + 1) * 4, len_bytes = static_cast<size_t>(B) * 4;
  const size_t pos_bytes = static_cast<size_t>(total_m) * 4;
  MAP_TRY(ensure(c->qoff, off_bytes + 2 * len_bytes));
  MAP_TRY(ensure(c->post, pos_bytes));
  {
    std::vector<long long> offs(B);
    long long acc = 0;
    for (int b = 0; b < B; ++b) { offs[b] = acc; acc += lens[b]; }
    int32_t* qo = static_cast<int32_t*>(c->qoff.p);
    CU_TRY(mapk::launch_query_meta(lens, offs.data(), B, N, qo, qo + (B + 1), static_cast<int32_t*>(c->post.p), nv,
                                   nv ? qo + (2 * B + 1) : nullptr, st));
    c->counters.launches += (B + 1023) / 1024;
  }
  const int* d_off = static_cast<const int*>(c->qoff.p);
  const int* d_len = d_off + (B + 1);
  const int* d_nv = nv ? d_off + (2 * B + 1) : nullptr;

  const long long vrows = static_cast<long long>(B) * N;
  const int dp3 = 3 * g.dp;
  MAP_TRY(ensure(c->kb, static_cast<size_t>(vrows) * dp3 * 2));
  MAP_TRY(ensure(c->qb, static_cast<size_t>(total_m) * dp3 * 2));
  MAP_TRY(ensure(c->h1, static_cast<size_t>(vrows) * g.Dh * 4));
  MAP_TRY(ensure(c->th1, static_cast<size_t>(total_m) * g.Dh * 4));
  const Modality mt{text, total_m, c->w[0], c->w[1], c->wqt, c->bqt, c->th1.p, c->qb.p, 1,
                    1.0f / std::sqrt(static_cast<float>(g.dp)), q_out, static_cast<const int*>(c->post.p), 1, nullptr, 0};
  const Modality mv{vis, vrows, c->w[5], c->w[6], c->wkv, c->bkv, c->h1.p, c->kb.p, 0, 1.0f, k_out, nullptr, N, d_nv, N};
  long long valid = vrows;
  if (nv) {
    valid = 0;
    for (int b = 0; b < B; ++b) valid += nv[b];
  }
  MAP_TRY(predictor(c, mv, mt, mapk::predictor_tile_width(valid, total_m, g.Dh, g.D, c->num_sms), st));
  // Eq. 3 on the tensor cores: logits tile [visual tokens x question tokens] of one image,
  // pass 1 -> per-slab column (max, sum exp), combine -> max + ln(sum), pass 2 -> mean.
  const int m_tiles = (N + 127) / 128, nparts = 4 * m_tiles;
  const int ld = ((max_m + 3) / 4) * 4;
  const int n_tiles = (max_m + 255) / 256;
  MAP_TRY(ensure(c->stats, static_cast<size_t>(B) * (nparts + 1) * ld * 8));
  float2* part = static_cast<float2*>(c->stats.p);
  float2* fin = part + static_cast<size_t>(B) * nparts * ld;
  GemmDesc d{};
  d.A = c->kb.p; d.a_rows_total = vrows; d.a_row_stride = N;
  d.B = c->qb.p; d.b_rows_total = total_m; d.b_row_stride = 0; d.b_off = d_off;
  d.M = N; d.N = max_m; d.K = dp3; d.batch = B; d.n_limit = d_len; d.col_count = d_len;
  d.m_limit = d_nv;
  d.status = c->status;
  float* mean_out = scores;
  if (n_tiles > 1) {
    MAP_TRY(ensure(c->pmean, static_cast<size_t>(vrows) * n_tiles * 4));
    mean_out = static_cast<float*>(c->pmean.p);
  }
  {
    Timed t(c, st, MAP_K_SCORES);
    d.epi = mapk::EPI_SM_STATS; d.stats = part; d.stat_ld = ld;
    d.C = part; d.ldc = 4; d.c_batch_stride = 0;
    MAP_TRY(gemm(c, d, st));
    d.epi = mapk::EPI_SM_MEAN;
    // One tile a CTA and few statistics: each tile combines its columns' slabs itself while its MMAs run, a
    // launch less.  128 threads take up to 256 columns, so a thread reads the slabs of one column or two, in
    // sequence.  Calls with a launch of its own against in the tile (D = 4096): 20 slabs (N = 576), up to 128
    // question tokens, 155.3 -> 153.7 us, 16 images 249.0 -> 246.7; 24 slabs 154.7 -> 152.2; 32 slabs 157.0 ->
    // 156.9 with 16 tokens, 158.8 -> 159.2 with 128; 36 slabs 160.4 -> 161.6.  Two columns: 8 slabs 158.5 -> 156.9,
    // 20 slabs 157.3 -> 158.2, 32 slabs 162.4 -> 166.3.
    const int per_thread = nparts * (max_m > 128 ? 2 : 1);
    if (per_thread <= kCombineInTile && static_cast<long long>(B) * m_tiles * n_tiles <= c->num_sms) {
      d.stats = part; d.stat_parts = nparts;
    } else {
      ++c->counters.launches;
      CU_TRY(mapk::launch_stats_combine(part, B, nparts, ld, d_len, fin, st));
      d.stats = fin;
    }
    d.C = mean_out; d.ldc = 4; d.c_batch_stride = static_cast<long long>(N) * n_tiles;
    MAP_TRY(gemm(c, d, st));
    if (n_tiles > 1) {
      ++c->counters.launches;
      CU_TRY(mapk::launch_sum_tiles(mean_out, B, N, n_tiles, 256, d_len, scores, st));
    }
  }
  return MAP_OK;
}

template <typename T>
T* carve(char*& p, size_t n) {
  T* r = reinterpret_cast<T*>(p);
  p += ((n * sizeof(T) + 255) / 256) * 256;
  return r;
}

// nv as for score_impl: tokens at or past nv[b] are never retained (K <= every nv[b]).
// gather_out: where to compact the kept rows as well (nullptr: not); *gathered tells whether that was
// done.
int select_impl(map_ctx* c, const float* scores, const void* vis, const int32_t* nv, int B, int N, int K,
                int32_t* keep, int32_t* order, cudaStream_t st, void* gather_out = nullptr, bool* gathered = nullptr) {
  if (!c || !scores || !vis) return MAP_EINVAL;
  if (B < 1 || N < 1 || K < 0 || K > N) return MAP_EINVAL;
  if (nv)
    for (int b = 0; b < B; ++b)
      if (nv[b] < 1 || nv[b] > N || K > nv[b]) return MAP_EINVAL;
  if (K == 0) return MAP_OK;
  if (!keep) return MAP_EINVAL;
  if (K > kMaxK || N > kMaxN) return MAP_EUNSUPPORTED;
  if (!aligned16(vis)) return MAP_EINVAL;
  CU_TRY(cudaSetDevice(c->device));
  Timed timed(c, st, MAP_K_SELECT);
  if (K == N) {
    ++c->counters.launches;
    CU_TRY(mapk::launch_sel_identity(B, N, keep, order, st));
    return MAP_OK;
  }
  const map_config& g = c->cfg;
  int K0 = resolve_k0(g, K);
  if (g.lambda == 0.f) K0 = K;        // values are p_hat alone: plain top-K
  if (K0 < K && K > kMaxKDiverse) return MAP_EUNSUPPORTED;
  const long long BN = static_cast<long long>(B) * N;
  const int S = mapk::kActiveSlots, R = ((S + K + 15) / 16) * 16;   // row stride of Vg and G (16-byte rows)

  mapk::SelState s{};
  const int KP = ((K + 3) / 4) * 4;
  s.B = B; s.N = N; s.D = g.D; s.K = K; s.K0 = K0; s.S = S; s.R = R; s.KP = KP;
  s.lambda = g.lambda; s.tau = g.tau;
  s.scores = scores; s.V = vis; s.status = c->status;
  if (nv) {                                      // valid tokens per image, on the device
    MAP_TRY(ensure(c->snv, static_cast<size_t>(B) * 4));
    c->counters.launches += (B + 2047) / 2048;
    CU_TRY(mapk::launch_put_ints(nv, B, static_cast<int32_t*>(c->snv.p), st));
    s.nvalid = static_cast<const int32_t*>(c->snv.p);
  }
  // per-token arrays
  MAP_TRY(ensure(c->sqn, BN * 4));
  MAP_TRY(ensure(c->sU, BN * 4));
  MAP_TRY(ensure(c->sr2, BN * 4));
  MAP_TRY(ensure(c->scstep, BN * 4));
  MAP_TRY(ensure(c->sstate, BN));
  MAP_TRY(ensure(c->spicks, static_cast<size_t>(B) * K * 4));
  MAP_TRY(ensure(c->sr0, static_cast<size_t>(B) * K * 4));
  MAP_TRY(ensure(c->sbt, static_cast<size_t>(B) * K * 4));
  MAP_TRY(ensure(c->srn, static_cast<size_t>(B) * K * 4));
  MAP_TRY(ensure(c->ssmall, static_cast<size_t>(B) * 4 * 16 + 24 * 256));
  static_assert(mapk::kReprojMax <= kProjMaxBasis, "re-projection basis limit");
  MAP_TRY(ensure(c->stheta, static_cast<size_t>(B) * 8));
  MAP_TRY(ensure(c->saslot, static_cast<size_t>(B) * S * 4));
  s.sqn = static_cast<float*>(c->sqn.p);
  s.U = static_cast<float*>(c->sU.p);
  s.r2 = static_cast<float*>(c->sr2.p);
  s.cstep = static_cast<int32_t*>(c->scstep.p);
  s.state = static_cast<uint8_t*>(c->sstate.p);
  s.picks = static_cast<int32_t*>(c->spicks.p);
  s.r0 = static_cast<int32_t*>(c->sr0.p);
  s.basis_tok = static_cast<int32_t*>(c->sbt.p);
  s.rnorm = static_cast<float*>(c->srn.p);
  char* sm = static_cast<char*>(c->ssmall.p);
  s.npicks = carve<int32_t>(sm, B);
  s.nbasis = carve<int32_t>(sm, B);
  s.done = carve<int32_t>(sm, B);
  s.mode = carve<int32_t>(sm, B);
  s.gbase = carve<int32_t>(sm, B);
  s.proj_lim = carve<int32_t>(sm, B);
  s.blist = carve<int32_t>(sm, B);
  s.bcount = carve<int32_t>(sm, 2);
  s.done_count = carve<int32_t>(sm, 1);
  s.uptr = carve<const void*>(sm, 2);
  int32_t* loop_iters = carve<int32_t>(sm, 1);
  s.theta = static_cast<uint64_t*>(c->stheta.p);
  s.aslot = static_cast<int32_t*>(c->saslot.p);

  // With 0 < K0 < K, one tensor-core pass over V after the first R0 tokens gives every
  // candidate its exact value on their basis (and ||v||^2); otherwise values start from
  // p_hat * ||v||^lambda.  The first K0c <= min(kCholMax, S) tokens of R0 are factored before the
  // pass, which takes their first 128 basis vectors; the rest of R0 is retained in the rounds after
  // it, as forced picks.  Where the basis has more vectors than the pass took, every value it gave
  // stays a valid upper bound (values only shrink as the basis grows).
  const int K0c = std::min({K0, mapk::kCholMax, S});
  const bool project = K0 > 0 && K0 < K;
  if (K0 < K && !project) {
    ++c->counters.launches;
    CU_TRY(mapk::launch_row_sqnorm(vis, BN, g.D, static_cast<float*>(c->sqn.p), st));
  } else if (K0 >= K) {
    CU_TRY(cudaMemsetAsync(c->sqn.p, 0, BN * 4, st));
  }
  ++c->counters.launches;
  {
    mapk::SelState si = s;
    if (project) si.sqn = nullptr;     // written by the projection
    CU_TRY(mapk::launch_sel_init(si, st));
  }
  if (K0 < K) {
    MAP_TRY(ensure(c->sEc, static_cast<size_t>(BN) * KP * 4));
    MAP_TRY(ensure(c->sVg, static_cast<size_t>(B) * R * g.D * 2));
    MAP_TRY(ensure(c->sG, static_cast<size_t>(B) * S * R * 4));
    s.Ec = static_cast<float*>(c->sEc.p);
    s.Vg = c->sVg.p;
    s.G = static_cast<float*>(c->sG.p);
    // the GEMM after a list producer reads the count that producer appended through
    auto take_list = [&](GemmDesc& g) { g.bcount = s.bcount + s.bc_par; s.bc_par ^= 1; };
    // Rounds: every round picks or makes S stale bounds exact, so at most ceil(N / S) rounds
    // without a pick come before each pick; one more per kRoundPicks picks of a launch.
    const long long cap = static_cast<long long>(K) * ((N + S - 1) / S + 1) +
                          (K + mapk::kRoundPicks - 1) / mapk::kRoundPicks + 64;
    if (project) {
      // R0: G[R0, R0] on the tensor cores, then its Cholesky factor.
      c->counters.launches += 3;
      CU_TRY(mapk::launch_sel_choose(s, st));
      CU_TRY(mapk::launch_sel_gram(s, K0c, 0, c->wait_ns, st));
      {
        mapk::SelState sc = s;        // the first K0c tokens of R0
        sc.K0 = K0c;
        CU_TRY(mapk::launch_sel_chol(sc, st));
      }
      ++c->counters.select_rounds;
      // every candidate's exact value: one tensor-core pass over V against the R0 basis
      GemmDesc pd{};
      pd.A = vis; pd.a_rows_total = BN; pd.a_row_stride = N;
      pd.B = s.Vg; pd.b_rows_total = static_cast<long long>(B) * R; pd.b_row_stride = R; pd.b_base = S;
      pd.M = N; pd.N = kProjMaxBasis; pd.K = g.D; pd.batch = B; pd.n_limit = s.proj_lim;
      pd.blist = s.blist;                         // images to project (built by the gather)
      pd.m_limit = s.nvalid;
      pd.C = nullptr; pd.ldc = 0; pd.c_batch_stride = 0;
      pd.epi = mapk::EPI_PROJECT; pd.status = c->status;
      pd.proj.state = s.state; pd.proj.scores = scores; pd.proj.Ec = s.Ec; pd.proj.KP = KP;
      pd.proj.basis_tok = s.basis_tok; pd.proj.rnorm = s.rnorm; pd.proj.nbasis = s.nbasis; pd.proj.Kcap = K;
      pd.proj.lambda = g.lambda; pd.proj.tau = g.tau;
      pd.proj.r2 = s.r2; pd.proj.U = s.U; pd.proj.sqn = static_cast<float*>(c->sqn.p); pd.proj.cstep = s.cstep;
      auto project_all = [&](bool first) -> int {
        ++c->counters.launches;
        CU_TRY(mapk::launch_sel_gather(s, first, st));
        take_list(pd);
        return gemm(c, pd, st);
      };
      // Basis columns a projection on n vectors computes: 32 for the smallest R0 (one image of 576 tokens,
      // k = 32: 1.014 times faster than with 96).  64 for 33 to 64 vectors is not built; measured in a copy it took
      // 184 -> 181 us for one image of 576 tokens and k = 96, 212 -> 210 us of 2880.
      auto proj_cols = [](int n) { return n <= 32 ? 32 : (n <= 96 ? 96 : kProjMaxBasis); };
      pd.N = proj_cols(K0c);
      MAP_TRY(project_all(true));
      pd.N = proj_cols(K);
      // One round (greedy, or the rest of R0 when K0 > K0c).  After a projection on the whole of R0's
      // basis every coordinate is current; then the images still selecting are projected again on
      // their whole basis (when it has at most kReprojMax vectors): exact values for every candidate
      // make the next active set the true top S.
      const bool whole = K0c <= mapk::kReprojMax;
      c->counters.launches += whole ? 4 : 5;
      CU_TRY(mapk::launch_sel_choose(s, st));
      CU_TRY(mapk::launch_sel_gram(s, S, std::max(0, K0c - mapk::kReprojMax), c->wait_ns, st));
      CU_TRY(mapk::launch_sel_greedy(s, !whole, st));
      ++c->counters.select_rounds;
      if (whole) MAP_TRY(project_all(false));
    }
    // The remaining rounds run as a device-side loop (a CUDA graph whose WHILE node repeats a
    // round while an image still selects): the host never waits for them.
    if (!c->loops) c->loops = mapk::sel_loop_cache_create();
    if (!c->loops) return MAP_ENOMEM;
    ++c->counters.launches;            // the test kernel ahead of the loop; iterations are counted on the device
    CU_TRY(mapk::launch_sel_loop(c->loops, s, c->wait_ns, static_cast<int>(cap), loop_iters, c->loop_iters_total, st));
  } else {
    ++c->counters.launches;
    CU_TRY(mapk::launch_sel_copy_r0(s.r0, B, K, s.picks, st));
  }
  ++c->counters.launches;
  if (gather_out && !order && !c->timing && K <= mapk::kFinalizeGatherMax && 2 * K <= g.D && B <= 65535 &&
      aligned16(vis) && aligned16(gather_out)) {
    CU_TRY(mapk::launch_sel_finalize_gather(s.picks, B, K, vis, N, g.D, keep, gather_out, c->status, st));
    *gathered = true;
    return MAP_OK;
  }
  CU_TRY(mapk::launch_sel_finalize(s.picks, B, K, keep, order, st));
  return MAP_OK;
}

int gather_impl(map_ctx* c, const void* vis, const int32_t* keep, int B, int N, int K, void* out, cudaStream_t st) {
  if (!c || !vis) return MAP_EINVAL;
  if (B < 1 || N < 1 || K < 0) return MAP_EINVAL;
  if (K == 0) return MAP_OK;
  if (!keep || !out) return MAP_EINVAL;
  if (!aligned16(vis) || !aligned16(out)) return MAP_EINVAL;
  CU_TRY(cudaSetDevice(c->device));
  Timed t(c, st, MAP_K_GATHER);
  ++c->counters.launches;
  CU_TRY(mapk::launch_gather(vis, keep, B, N, K, c->cfg.D, out, c->status, st));
  return MAP_OK;
}

int assemble_impl(map_ctx* ctx, const void* vis_feats, const int32_t* keep_idx, const void* text_feats,
                  const int32_t* lens, const int32_t* nv, int B, int N, int k, int pos_offset, void* seq,
                  int32_t* pos_ids, cudaStream_t st) {
  if (!ctx || !vis_feats || !text_feats || !lens) return MAP_EINVAL;
  if (B < 1 || N < 1 || k < 0 || k > N) return MAP_EINVAL;
  long long rows = 0;
  for (int b = 0; b < B; ++b) {
    if (lens[b] < 0) return MAP_EINVAL;
    if (nv && (nv[b] < 1 || nv[b] > N || k > nv[b])) return MAP_EINVAL;
    rows += k + lens[b];
  }
  if (rows == 0) return MAP_OK;
  if (!seq || !pos_ids || (k > 0 && !keep_idx)) return MAP_EINVAL;
  if (!aligned16(vis_feats) || !aligned16(text_feats) || !aligned16(seq)) return MAP_EINVAL;
  CU_TRY(cudaSetDevice(ctx->device));
  ++ctx->counters.launches;
  CU_TRY(mapk::launch_assemble(vis_feats, keep_idx, text_feats, lens, nv, B, N, k, ctx->cfg.D, pos_offset, seq,
                               pos_ids, ctx->status, st));
  return MAP_OK;
}

bool is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

// Read-only view of a context for other translation units of the library.
namespace mapk {
struct CtxView {
  const map_config* cfg;
  int device, num_sms;
  int* status;
  int32_t* h_done;
  long long* launches;
  long long* rounds;
  int* h_status;
  int32_t* h_done_dev;
  int* h_status_dev;
  int* deferred;
};
CtxView ctx_view(map_ctx* c) {
  return CtxView{&c->cfg, c->device, c->num_sms, c->status, c->h_done, &c->counters.launches,
                 &c->counters.select_rounds, c->h_status, c->h_done_dev, c->h_status_dev, &c->deferred};
}
}  // namespace mapk

extern "C" {

int map_config_default(map_config* cfg) {
  if (!cfg) return MAP_EINVAL;
  cfg->D = 4096; cfg->Dh = 1024; cfg->dp = 128;
  cfg->rope_theta = 10000.f; cfg->rope_on = 1;
  cfg->k0_frac = 0.5f; cfg->k0_abs = -1;
  cfg->lambda = 1.0f; cfg->tau = 1e-5f;
  return MAP_OK;
}

int map_init(const map_config* cfg, const map_weights* w, map_ctx** out) {
  if (!out) return MAP_EINVAL;
  *out = nullptr;
  if (check_config(cfg) != MAP_OK || !w) return MAP_EINVAL;
  const void* src[10] = {w->wT1, w->bT1, w->wT2, w->bT2, w->wQ, w->wV1, w->bV1, w->wV2, w->bV2, w->wK};
  for (const void* p : src)
    if (!p) return MAP_EINVAL;
  map_ctx* c = new (std::nothrow) map_ctx();
  if (!c) return MAP_ENOMEM;
  c->cfg = *cfg;
  int rc = MAP_OK;
  do {
    if (cudaGetDevice(&c->device) != cudaSuccess) { rc = MAP_ECUDA; break; }
    if (cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) { rc = MAP_ECUDA; break; }
    const size_t D = cfg->D, Dh = cfg->Dh, dp = cfg->dp;
    const size_t rows[10] = {Dh, 1, Dh, 1, dp, Dh, 1, Dh, 1, dp};
    const size_t cols[10] = {D, Dh, Dh, Dh, Dh, D, Dh, Dh, Dh, Dh};
    for (int i = 0; i < 10 && rc == MAP_OK; ++i) {
      if (cudaMalloc(&c->w[i], rows[i] * cols[i] * 2) != cudaSuccess) { rc = MAP_ENOMEM; break; }
      if (cudaMemcpy(c->w[i], src[i], rows[i] * cols[i] * 2, cudaMemcpyDefault) != cudaSuccess) rc = MAP_ECUDA;
    }
    if (rc != MAP_OK) break;
    // The projections follow the second MLP layers with nothing in between: fold them.
    if (cudaMalloc(&c->wqt, dp * 3 * Dh * 2) != cudaSuccess || cudaMalloc(&c->wkv, dp * 3 * Dh * 2) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&c->bqt), dp * 4) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&c->bkv), dp * 4) != cudaSuccess) {
      rc = MAP_ENOMEM;
      break;
    }
    if (mapk::launch_fold_weights(c->w[4], c->w[2], c->w[3], static_cast<int>(dp), static_cast<int>(Dh), c->wqt,
                                  c->bqt, nullptr) != cudaSuccess ||
        mapk::launch_fold_weights(c->w[9], c->w[7], c->w[8], static_cast<int>(dp), static_cast<int>(Dh), c->wkv,
                                  c->bkv, nullptr) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess) {
      rc = MAP_ECUDA;
      break;
    }
    if (cudaMalloc(reinterpret_cast<void**>(&c->loop_iters_total), sizeof(long long)) != cudaSuccess) {
      rc = MAP_ENOMEM;
      break;
    }
    if (cudaMemset(c->loop_iters_total, 0, sizeof(long long)) != cudaSuccess) { rc = MAP_ECUDA; break; }
    if (cudaMalloc(&c->status, sizeof(int)) != cudaSuccess) { rc = MAP_ENOMEM; break; }
    if (cudaMemset(c->status, 0, sizeof(int)) != cudaSuccess) { rc = MAP_ECUDA; break; }
    if (cudaHostAlloc(&c->h_status, sizeof(int), cudaHostAllocMapped) != cudaSuccess) { rc = MAP_ENOMEM; break; }
    if (cudaHostAlloc(&c->h_done, sizeof(int32_t), cudaHostAllocMapped) != cudaSuccess) { rc = MAP_ENOMEM; break; }
    if (cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->h_status_dev), c->h_status, 0) != cudaSuccess ||
        cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->h_done_dev), c->h_done, 0) != cudaSuccess) {
      rc = MAP_ECUDA;
      break;
    }
  } while (false);
  if (rc != MAP_OK) {
    cudaGetLastError();
    map_destroy(c);
    return rc;
  }
  *out = c;
  return MAP_OK;
}

int map_score(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens, int B, int N,
              float* scores, void* stream) {
  return score_impl(ctx, text_feats, vis_feats, lens, nullptr, B, N, scores, nullptr, nullptr,
                    static_cast<cudaStream_t>(stream));
}

int map_score_debug(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens, int B, int N,
                    float* scores, float* q_out, float* k_out, void* stream) {
  return score_impl(ctx, text_feats, vis_feats, lens, nullptr, B, N, scores, q_out, k_out,
                    static_cast<cudaStream_t>(stream));
}

int map_select(map_ctx* ctx, const float* scores, const void* vis_feats, int B, int N, int k, int32_t* keep_idx,
               int32_t* pick_order, void* stream) {
  return select_impl(ctx, scores, vis_feats, nullptr, B, N, k, keep_idx, pick_order,
                     static_cast<cudaStream_t>(stream));
}

int map_gather(map_ctx* ctx, const void* vis_feats, const int32_t* keep_idx, int B, int N, int k, void* out,
               void* stream) {
  return gather_impl(ctx, vis_feats, keep_idx, B, N, k, out, static_cast<cudaStream_t>(stream));
}

int map_assemble(map_ctx* ctx, const void* vis_feats, const int32_t* keep_idx, const void* text_feats,
                 const int32_t* lens, int B, int N, int k, int pos_offset, void* seq, int32_t* pos_ids,
                 void* stream) {
  return assemble_impl(ctx, vis_feats, keep_idx, text_feats, lens, nullptr, B, N, k, pos_offset, seq, pos_ids,
                       static_cast<cudaStream_t>(stream));
}

int map_assemble_ragged(map_ctx* ctx, const void* vis_feats, const int32_t* keep_idx, const void* text_feats,
                        const int32_t* lens, const int32_t* n_valid, int B, int N, int k, int pos_offset, void* seq,
                        int32_t* pos_ids, void* stream) {
  if (!n_valid) return MAP_EINVAL;
  return assemble_impl(ctx, vis_feats, keep_idx, text_feats, lens, n_valid, B, N, k, pos_offset, seq, pos_ids,
                       static_cast<cudaStream_t>(stream));
}

}  // extern "C"

namespace {
int prune_impl(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens, const int32_t* nv,
               int B, int N, int k, void* out, int32_t* keep_idx, float* scores, void* stream) {
  if (!ctx || !text_feats || !vis_feats || !lens || !out || !keep_idx) return MAP_EINVAL;
  if (B < 1 || N < 1 || k < 0 || k > N) return MAP_EINVAL;
  if (nv)
    for (int b = 0; b < B; ++b)
      if (nv[b] < 1 || nv[b] > N || k > nv[b]) return MAP_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  map_ctx* c = ctx;
  CU_TRY(cudaSetDevice(c->device));
  long long total_m = 0;
  for (int b = 0; b < B; ++b) {
    if (lens[b] < 1) return MAP_EINVAL;
    total_m += lens[b];
  }
  const size_t D = c->cfg.D;
  const size_t vis_bytes = static_cast<size_t>(B) * N * D * 2, text_bytes = static_cast<size_t>(total_m) * D * 2;
  const size_t out_bytes = static_cast<size_t>(B) * k * D * 2, keep_bytes = static_cast<size_t>(B) * k * 4;
  const size_t sc_bytes = static_cast<size_t>(B) * N * 4;
  const bool dv = is_device_ptr(vis_feats), dt = is_device_ptr(text_feats), dout = is_device_ptr(out);
  const bool dkeep = is_device_ptr(keep_idx), dsc = scores ? is_device_ptr(scores) : true;
  const void* v = vis_feats;
  const void* t = text_feats;
  if (!dv) { MAP_TRY(ensure(c->pvis, vis_bytes)); v = c->pvis.p; }
  if (!dt) { MAP_TRY(ensure(c->ptext, text_bytes)); t = c->ptext.p; }
  void* o = out;
  int32_t* kp = keep_idx;
  float* sp = scores;
  if (!dout) { MAP_TRY(ensure(c->pout, out_bytes)); o = c->pout.p; }
  if (!dkeep) { MAP_TRY(ensure(c->pkeep, keep_bytes)); kp = static_cast<int32_t*>(c->pkeep.p); }
  if (!dsc || !scores) { MAP_TRY(ensure(c->pscores, sc_bytes)); sp = static_cast<float*>(c->pscores.p); }
  const bool host_io = !dv || !dt || !dout || !dkeep || (scores && !dsc);

  // With host buffers the batch runs as a pipeline of image chunks: chunk i+1 is copied in
  // (stream s_in) while chunk i is scored, selected and gathered (the caller's stream) and
  // chunk i-1 is copied out (stream s_out).  Results equal the one-shot path.
  const int nchunk = host_io ? std::min(B, 4) : 1;
  if (nchunk > 1) {
    if (!c->s_in) CU_TRY(cudaStreamCreateWithFlags(&c->s_in, cudaStreamNonBlocking));
    if (!c->s_out) CU_TRY(cudaStreamCreateWithFlags(&c->s_out, cudaStreamNonBlocking));
  }
  std::vector<long long> toff(B + 1, 0);
  for (int b = 0; b < B; ++b) toff[b + 1] = toff[b] + lens[b];
  cudaStream_t si = nchunk > 1 ? c->s_in : st, so = nchunk > 1 ? c->s_out : st;
  std::vector<cudaEvent_t> evs;
  auto ev = [&]() { cudaEvent_t e = take_event(c); evs.push_back(e); return e; };
  auto finish = [&](int rc) {
    for (cudaEvent_t e : evs) c->free_events.push_back(e);
    return rc;
  };
  if (nchunk > 1) {                         // buffers reused from earlier work on the caller's stream
    cudaEvent_t e0 = ev();
    if (cudaEventRecord(e0, st) != cudaSuccess || cudaStreamWaitEvent(si, e0, 0) != cudaSuccess ||
        cudaStreamWaitEvent(so, e0, 0) != cudaSuccess)
      return finish(MAP_ECUDA);
  }
  std::vector<cudaEvent_t> ev_in(nchunk);
  // Chunk boundaries, weights 3 : 3 : ... : 1.  The copy engine idles from the end of the last
  // copy-in until the call returns, i.e. while the last chunk is scored, selected, gathered and
  // copied out, so the last chunk is the small one; the others stay copy-bound.
  std::vector<int> cb(nchunk + 1, 0);
  {
    const int wsum = 3 * (nchunk - 1) + 1;
    for (int i = 1; i < nchunk; ++i) {
      const int v = static_cast<int>(static_cast<long long>(B) * 3 * i / wsum);
      cb[i] = std::min(std::max(v, cb[i - 1] + 1), B - (nchunk - i));
    }
    cb[nchunk] = B;
  }
  auto chunk = [&](int i, int& b0, int& b1) { b0 = cb[i]; b1 = cb[i + 1]; };
  for (int i = 0; i < nchunk; ++i) {
    int b0, b1;
    chunk(i, b0, b1);
    const size_t vo = static_cast<size_t>(b0) * N * D * 2, vn = static_cast<size_t>(b1 - b0) * N * D * 2;
    const size_t to = static_cast<size_t>(toff[b0]) * D * 2, tn = static_cast<size_t>(toff[b1] - toff[b0]) * D * 2;
    if (!dv && cudaMemcpyAsync(static_cast<char*>(c->pvis.p) + vo, static_cast<const char*>(vis_feats) + vo, vn,
                               cudaMemcpyHostToDevice, si) != cudaSuccess)
      return finish(MAP_ECUDA);
    if (!dt && cudaMemcpyAsync(static_cast<char*>(c->ptext.p) + to, static_cast<const char*>(text_feats) + to, tn,
                               cudaMemcpyHostToDevice, si) != cudaSuccess)
      return finish(MAP_ECUDA);
    ev_in[i] = ev();
    if (cudaEventRecord(ev_in[i], si) != cudaSuccess) return finish(MAP_ECUDA);
  }
  for (int i = 0; i < nchunk; ++i) {
    int b0, b1;
    chunk(i, b0, b1);
    const int Bc = b1 - b0;
    if (cudaStreamWaitEvent(st, ev_in[i], 0) != cudaSuccess) return finish(MAP_ECUDA);
    const void* vc = static_cast<const char*>(v) + static_cast<size_t>(b0) * N * D * 2;
    const void* tc = static_cast<const char*>(t) + static_cast<size_t>(toff[b0]) * D * 2;
    float* spc = sp + static_cast<size_t>(b0) * N;
    int32_t* kpc = kp + static_cast<size_t>(b0) * k;
    void* oc = static_cast<char*>(o) + static_cast<size_t>(b0) * k * D * 2;
    const int32_t* nvc = nv ? nv + b0 : nullptr;
    int rc = score_impl(c, tc, vc, lens + b0, nvc, Bc, N, spc, nullptr, nullptr, st);
    bool gathered = false;
    if (rc == MAP_OK) rc = select_impl(c, spc, vc, nvc, Bc, N, k, kpc, nullptr, st, oc, &gathered);
    if (rc == MAP_OK && !gathered) rc = gather_impl(c, vc, kpc, Bc, N, k, oc, st);
    if (rc != MAP_OK) return finish(rc);
    if (host_io) {
      cudaEvent_t ed = ev();
      if (cudaEventRecord(ed, st) != cudaSuccess || cudaStreamWaitEvent(so, ed, 0) != cudaSuccess) return finish(MAP_ECUDA);
      const size_t oo = static_cast<size_t>(b0) * k * D * 2, on = static_cast<size_t>(Bc) * k * D * 2;
      const size_t ko = static_cast<size_t>(b0) * k * 4, kn = static_cast<size_t>(Bc) * k * 4;
      const size_t so_ = static_cast<size_t>(b0) * N * 4, sn = static_cast<size_t>(Bc) * N * 4;
      if (!dout && on && cudaMemcpyAsync(static_cast<char*>(out) + oo, static_cast<char*>(o) + oo, on,
                                         cudaMemcpyDeviceToHost, so) != cudaSuccess)
        return finish(MAP_ECUDA);
      if (!dkeep && kn && cudaMemcpyAsync(reinterpret_cast<char*>(keep_idx) + ko, reinterpret_cast<char*>(kp) + ko, kn,
                                          cudaMemcpyDeviceToHost, so) != cudaSuccess)
        return finish(MAP_ECUDA);
      if (scores && !dsc && cudaMemcpyAsync(reinterpret_cast<char*>(scores) + so_, reinterpret_cast<char*>(sp) + so_,
                                            sn, cudaMemcpyDeviceToHost, so) != cudaSuccess)
        return finish(MAP_ECUDA);
    }
  }
  if (host_io) {
    if (nchunk > 1) {
      cudaEvent_t ee = ev();
      if (cudaEventRecord(ee, so) != cudaSuccess || cudaStreamWaitEvent(st, ee, 0) != cudaSuccess) return finish(MAP_ECUDA);
    }
    if (cudaStreamSynchronize(st) != cudaSuccess) return finish(MAP_ECUDA);
  }
  return finish(MAP_OK);
}
}  // namespace

extern "C" {

int map_prune(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens, int B, int N, int k,
              void* out, int32_t* keep_idx, float* scores, void* stream) {
  return prune_impl(ctx, text_feats, vis_feats, lens, nullptr, B, N, k, out, keep_idx, scores, stream);
}

int map_prune_ragged(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens,
                     const int32_t* n_valid, int B, int N, int k, void* out, int32_t* keep_idx, float* scores,
                     void* stream) {
  if (!n_valid) return MAP_EINVAL;
  return prune_impl(ctx, text_feats, vis_feats, lens, n_valid, B, N, k, out, keep_idx, scores, stream);
}

int map_score_ragged(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens,
                     const int32_t* n_valid, int B, int N, float* scores, void* stream) {
  if (!n_valid) return MAP_EINVAL;
  return score_impl(ctx, text_feats, vis_feats, lens, n_valid, B, N, scores, nullptr, nullptr,
                    static_cast<cudaStream_t>(stream));
}

int map_select_ragged(map_ctx* ctx, const float* scores, const void* vis_feats, const int32_t* n_valid, int B, int N,
                      int k, int32_t* keep_idx, int32_t* pick_order, void* stream) {
  if (!n_valid) return MAP_EINVAL;
  return select_impl(ctx, scores, vis_feats, n_valid, B, N, k, keep_idx, pick_order,
                     static_cast<cudaStream_t>(stream));
}

int map_distill_grad(map_ctx* ctx, const void* text_feats, const void* vis_feats, const int32_t* lens,
                     const float* teacher, int B, int N, float* loss, const map_grads* grads, void* stream) {
  if (!ctx || !text_feats || !vis_feats || !lens || !teacher || !loss || !grads) return MAP_EINVAL;
  float* gout[10] = {grads->wT1, grads->bT1, grads->wT2, grads->bT2, grads->wQ,
                     grads->wV1, grads->bV1, grads->wV2, grads->bV2, grads->wK};
  for (float* p : gout)
    if (!p) return MAP_EINVAL;
  if (B < 1 || N < 1) return MAP_EINVAL;
  long long total_m = 0;
  int max_m = 0;
  for (int b = 0; b < B; ++b) {
    if (lens[b] < 1) return MAP_EINVAL;
    total_m += lens[b];
    max_m = std::max(max_m, static_cast<int>(lens[b]));
  }
  if (total_m > (1ll << 24) || static_cast<long long>(B) * N > (1ll << 24)) return MAP_EUNSUPPORTED;
  map_ctx* c = ctx;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const map_config& g = c->cfg;
  const long long D = g.D, Dh = g.Dh, dp = g.dp, Tv = static_cast<long long>(B) * N, Tt = total_m;
  CU_TRY(cudaSetDevice(c->device));
  MAP_TRY(ensure_rope(c, g.rope_on ? N + max_m + 1 : 1));
  // the most rows a training step takes (the elementwise kernels' grids, 64 rows a block, hold twice that)
  if ((std::max(Tv, Tt) + 31) / 32 > 65535) return MAP_EUNSUPPORTED;
  // question offsets and positions N + m (as for map_score)
  MAP_TRY(ensure(c->qoff, static_cast<size_t>(3 * B + 1) * 4));
  MAP_TRY(ensure(c->post, static_cast<size_t>(total_m) * 4));
  std::vector<long long> offs(B);
  long long prows = 0;                               // question rows, each image's padded to 64
  {
    long long acc = 0;
    for (int b = 0; b < B; ++b) {
      offs[b] = acc;
      acc += lens[b];
      prows += (lens[b] + 63) / 64 * 64;
    }
  }
  int32_t* qo = static_cast<int32_t*>(c->qoff.p);
  int32_t* d_len = qo + (B + 1);
  int32_t* post = static_cast<int32_t*>(c->post.p);
  long long launches = (B + 1023) / 1024;
  CU_TRY(mapk::launch_query_meta(lens, offs.data(), B, N, qo, d_len, post, nullptr, nullptr, st));

  const int nblk = (N + 255) / 256, iN = N, iD = g.D, iDh = g.Dh, idp = g.dp;
  const long long Np = (N + 3) / 4 * 4;              // logits row stride: 16-byte aligned rows
  const int Nk = (N + 63) / 64 * 64;                 // columns of a staged logits term
  const float rs = 1.0f / std::sqrt(static_cast<float>(dp));
  const float2* tab = static_cast<const float2*>(c->rope.p);
  // The modalities meet only in Eq. 3 and its gradient: the question branch, a chain of launches
  // too small to fill the GPU, runs on a second stream beside the visual one, forward and backward
  // (4 samples of 2880 tokens: 922 -> 805 us, 2 of 576: 374 -> 253 us).
  MAP_TRY(ensure_aux(c));
  auto after = [&](cudaStream_t first, cudaStream_t then, cudaEvent_t e) -> int {
    CU_TRY(cudaEventRecord(e, first));
    return cuda_err(cudaStreamWaitEvent(then, e, 0));
  };
  // One modality: its rows, weights (first index, projection), buffers and stream.
  struct Branch {
    long long T; const void* X; int i1, ip; cudaStream_t st;
    const int32_t* pos; int pos_mod;
    const void* xa;                                  // the features, 16-byte aligned
    float *g1, *raw, *pre, *part, *ws;               // g1: GELU'(z1)
    uint16_t *h1, *h2, *dpre, *dh2, *dh1;
    long long ws_floats;
  };
  Branch br[2] = {};
  br[0].T = Tv; br[0].X = vis_feats; br[0].i1 = 5; br[0].ip = 9; br[0].st = st;
  br[0].pos = nullptr; br[0].pos_mod = g.rope_on ? N : 1;
  br[1].T = Tt; br[1].X = text_feats; br[1].i1 = 0; br[1].ip = 4; br[1].st = c->s_aux;
  br[1].pos = g.rope_on ? post : nullptr; br[1].pos_mod = 1;
  const int ks_dq = mapk::tc_ksplit(max_m, idp, iN, 6, c->num_sms);
  auto slices = [&](long long M, int Nn, long long K, int products) {
    return mapk::tc_ksplit(static_cast<int>(M), Nn, static_cast<int>(K), products, c->num_sms);
  };
  for (Branch& x : br) {                             // K slices of the branch's contractions
    const int T = static_cast<int>(x.T);
    auto need = [&](long long M, int Nn, long long K, int products) {
      const int ks = slices(M, Nn, K, products);
      if (ks > 1) x.ws_floats = std::max(x.ws_floats, ks * M * ((Nn + 3) / 4 * 4));
    };
    need(T, iDh, D, 1); need(T, iDh, Dh, 3); need(T, idp, Dh, 3);
    need(dp, iDh, T, 6); need(T, iDh, dp, 3); need(Dh, iDh, T, 6); need(T, iDh, Dh, 3); need(Dh, iD, T, 3);
  }
  // workspace: carved twice, first for its size
  float *S = nullptr, *dq = nullptr, *dk = nullptr, *p_hat = nullptr, *gb = nullptr, *part = nullptr,
        *ws_dq = nullptr;
  uint16_t *kk = nullptr, *qq = nullptr, *dl = nullptr;
  int32_t *poff = nullptr, *prow = nullptr, *img = nullptr;
  size_t used = 0;
  auto carve_all = [&](char* base) {
    used = 0;
    auto take = [&](auto*& p, long long n) {
      using T = std::remove_reference_t<decltype(*p)>;
      p = reinterpret_cast<T*>(base + used);
      used += (static_cast<size_t>(n) * sizeof(T) + 255) / 256 * 256;
    };
    for (Branch& x : br) {
      take(x.g1, x.T * Dh); take(x.raw, x.T * Dh); take(x.pre, x.T * dp);
      take(x.part, (x.T + 63) / 64 * Dh); take(x.ws, x.ws_floats);
      take(x.h1, x.T * 3 * Dh); take(x.h2, x.T * 3 * Dh); take(x.dh2, x.T * 3 * Dh); take(x.dh1, x.T * 3 * Dh);
      take(x.dpre, x.T * 3 * dp);
      uint16_t* xc = nullptr;
      x.xa = x.X;
      if (!aligned16(x.X)) { take(xc, x.T * D); x.xa = xc; }
    }
    take(kk, Tv * 3 * dp); take(qq, prows * 3 * dp);
    take(S, prows * Np); take(dl, prows * 3 * Nk);
    take(dq, prows * dp); take(ws_dq, ks_dq > 1 ? static_cast<long long>(ks_dq) * prows * dp : 0); take(dk, Tv * dp);
    take(p_hat, static_cast<long long>(B) * N); take(gb, static_cast<long long>(B) * N);
    take(part, static_cast<long long>(B) * nblk);
    take(poff, B); take(prow, total_m); take(img, prows);
  };
  carve_all(nullptr);
  MAP_TRY(ensure(c->dist, used));
  carve_all(static_cast<char*>(c->dist.p));

  using mapk::TcBatch; using mapk::TcOperand; using mapk::TcResult;
  auto split = [](const uint16_t* p, long long rows, int cols, int mn) { return TcOperand{p, rows, 3 * cols, cols, mn}; };
  auto exact = [](const void* p, long long rows, int cols, int mn) { return TcOperand{p, rows, cols, 0, mn}; };
  auto mm = [&](long long M, int Nn, long long K, const TcOperand& A, const TcOperand& Bo, const TcBatch& bt, int ks,
                bool add, float* C, long long ldc, float* ws, cudaStream_t s, TcResult* res) -> int {
    cudaError_t e = mapk::launch_tc_matmul(static_cast<int>(M), Nn, static_cast<int>(K), A, Bo, bt, ks, add, C, ldc, ws,
                                           c->num_sms, c->status, c->wait_ns, s, &launches, res);
    if (e == cudaErrorInvalidValue) return MAP_EUNSUPPORTED;
    return cuda_err(e);
  };
  ++launches;
  CU_TRY(mapk::launch_distill_meta(d_len, qo, B, poff, prow, img, st));
  // forward: z1 = X W1^T + b1, h1 = GELU(z1), h2 = h1 W2^T + b2, projection, RoPE
  auto forward = [&](const Branch& x, float scale, uint16_t* out, const int32_t* out_map) -> int {
    TcResult r;
    if (x.xa != x.X)
      CU_TRY(cudaMemcpyAsync(const_cast<void*>(x.xa), x.X, static_cast<size_t>(x.T) * D * 2, cudaMemcpyDeviceToDevice, x.st));
    MAP_TRY(mm(x.T, iDh, D, exact(x.xa, x.T, iD, 0), exact(c->w[x.i1], Dh, iD, 0), TcBatch{}, slices(x.T, iDh, D, 1),
               false, x.raw, Dh, x.ws, x.st, &r));
    CU_TRY(mapk::launch_act_split(true, r, c->w[x.i1 + 1], x.T, iDh, x.g1, x.h1, x.st));
    MAP_TRY(mm(x.T, iDh, Dh, split(x.h1, x.T, iDh, 0), exact(c->w[x.i1 + 2], Dh, iDh, 0), TcBatch{},
               slices(x.T, iDh, Dh, 3), false, x.raw, Dh, x.ws, x.st, &r));
    CU_TRY(mapk::launch_act_split(false, r, c->w[x.i1 + 3], x.T, iDh, nullptr, x.h2, x.st));
    MAP_TRY(mm(x.T, idp, Dh, split(x.h2, x.T, iDh, 0), exact(c->w[x.ip], dp, iDh, 0), TcBatch{},
               slices(x.T, idp, Dh, 3), false, x.pre, dp, x.ws, x.st, &r));
    CU_TRY(mapk::launch_rope_split(false, r, nullptr, x.T, idp, tab, c->rope_rows, x.pos, x.pos_mod, scale, out,
                                   out_map, x.st));
    launches += 3;
    return MAP_OK;
  };
  // backward through RoPE, the projection and the MLP
  auto backward = [&](const Branch& x, const TcResult& dpost, const int32_t* in_map, float scale) -> int {
    TcResult r;
    CU_TRY(mapk::launch_rope_split(true, dpost, in_map, x.T, idp, tab, c->rope_rows, x.pos, x.pos_mod, scale, x.dpre,
                                   nullptr, x.st));
    MAP_TRY(mm(dp, iDh, x.T, split(x.dpre, x.T, idp, 1), split(x.h2, x.T, iDh, 1), TcBatch{}, slices(dp, iDh, x.T, 6),
               true, gout[x.ip], Dh, x.ws, x.st, nullptr));                                          // dW_p
    MAP_TRY(mm(x.T, iDh, dp, split(x.dpre, x.T, idp, 0), exact(c->w[x.ip], dp, iDh, 1), TcBatch{},
               slices(x.T, iDh, dp, 3), false, x.raw, Dh, x.ws, x.st, &r));                          // dh2
    CU_TRY(mapk::launch_back_split(r, nullptr, x.T, iDh, x.dh2, x.part, gout[x.i1 + 3], x.st));
    MAP_TRY(mm(Dh, iDh, x.T, split(x.dh2, x.T, iDh, 1), split(x.h1, x.T, iDh, 1), TcBatch{}, slices(Dh, iDh, x.T, 6),
               true, gout[x.i1 + 2], Dh, x.ws, x.st, nullptr));                                      // dW2
    MAP_TRY(mm(x.T, iDh, Dh, split(x.dh2, x.T, iDh, 0), exact(c->w[x.i1 + 2], Dh, iDh, 1), TcBatch{},
               slices(x.T, iDh, Dh, 3), false, x.raw, Dh, x.ws, x.st, &r));                          // dh1
    CU_TRY(mapk::launch_back_split(r, x.g1, x.T, iDh, x.dh1, x.part, gout[x.i1 + 1], x.st));
    MAP_TRY(mm(Dh, iD, x.T, split(x.dh1, x.T, iDh, 1), exact(x.xa, x.T, iD, 1), TcBatch{}, slices(Dh, iD, x.T, 3), true,
               gout[x.i1], D, x.ws, x.st, nullptr));                                                 // dW1
    launches += 5;
    return MAP_OK;
  };
  auto step = [&]() -> int {
    MAP_TRY(after(st, c->s_aux, c->ev_fork));
    MAP_TRY(forward(br[1], rs, qq, prow));
    CU_TRY(mapk::launch_zero_pad_rows(qq, 3 * idp, img, prows, br[1].st));
    MAP_TRY(forward(br[0], 1.f, kk, nullptr));
    MAP_TRY(after(c->s_aux, st, c->ev_join));
    // Eq. 3 logits (q k / sqrt(dp), the scale is in q) of every image, softmax, KL, and dL/dlogits
    TcBatch lb;
    lb.n = B; lb.a_off = poff; lb.b_rows = iN; lb.m_count = d_len; lb.c_rows = prows;
    MAP_TRY(mm(max_m, iN, dp, split(qq, prows, idp, 0), split(kk, Tv, idp, 0), lb, 1, false, S, Np, nullptr, st, nullptr));
    CU_TRY(mapk::launch_distill_loss_grad(S, Np, prows, d_len, poff, img, teacher, B, N, p_hat, gb, part, loss, dl, Nk, st));
    launches += 5;
    // dk = dl^T q per image (K = its question rows, padded with zeros), dq = dl k (K = its tokens)
    TcResult rk, rq;
    TcBatch kb;
    kb.n = B; kb.a_off = poff; kb.b_off = poff; kb.k_count = d_len; kb.c_stride = static_cast<long long>(N) * dp;
    kb.c_rows = Tv;
    MAP_TRY(mm(N, idp, max_m, split(dl, prows, Nk, 1), split(qq, prows, idp, 1), kb, 1, false, dk, dp, nullptr, br[0].st, &rk));
    MAP_TRY(after(st, c->s_aux, c->ev_fork));
    TcBatch qb;
    qb.n = B; qb.a_off = poff; qb.b_rows = iN; qb.m_count = d_len; qb.c_rows = prows;
    MAP_TRY(mm(max_m, idp, N, split(dl, prows, Nk, 0), split(kk, Tv, idp, 1), qb, ks_dq, false, dq, dp, ws_dq, br[1].st, &rq));
    MAP_TRY(backward(br[1], rq, prow, rs));
    MAP_TRY(backward(br[0], rk, nullptr, 1.f));
    MAP_TRY(after(c->s_aux, st, c->ev_join));
    return MAP_OK;
  };
  const int rc = step();
  if (rc != MAP_OK) {                                // what the second stream still runs comes first
    after(c->s_aux, st, c->ev_join);
    return rc;
  }
  c->counters.launches += launches;
  return MAP_OK;
}

int map_status(map_ctx* ctx, void* stream) {
  if (!ctx) return MAP_EINVAL;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return MAP_ECUDA;
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return MAP_ECUDA;
  if (cudaMemcpy(ctx->h_status, ctx->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return MAP_ECUDA;
  int rc = dev_status_error(*ctx->h_status);
  if (*ctx->h_status) cudaMemset(ctx->status, 0, sizeof(int));
  if (rc == MAP_OK && ctx->deferred != MAP_OK) rc = ctx->deferred;
  ctx->deferred = MAP_OK;
  e = cudaGetLastError();
  if (rc == MAP_OK && e != cudaSuccess) rc = MAP_ECUDA;
  return rc;
}

void map_destroy(map_ctx* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  cudaDeviceSynchronize();
  for (void*& p : ctx->w)
    if (p) cudaFree(p);
  for (void* p : {ctx->wqt, ctx->wkv, static_cast<void*>(ctx->bqt), static_cast<void*>(ctx->bkv)})
    if (p) cudaFree(p);
  DevBuf* bufs[] = {&ctx->rope, &ctx->h1, &ctx->kb, &ctx->th1, &ctx->qb, &ctx->stats,
                    &ctx->qoff, &ctx->post, &ctx->sqn, &ctx->pmean, &ctx->snv, &ctx->dist, &ctx->sU, &ctx->sr2, &ctx->scstep, &ctx->sstate,
                    &ctx->sEc, &ctx->spicks, &ctx->sr0, &ctx->sbt, &ctx->srn, &ctx->ssmall, &ctx->stheta,
                    &ctx->saslot, &ctx->sVg, &ctx->sG, &ctx->pvis, &ctx->ptext, &ctx->pout, &ctx->pkeep,
                    &ctx->pscores};
  for (DevBuf* b : bufs) release(*b);
  if (ctx->status) cudaFree(ctx->status);
  if (ctx->loop_iters_total) cudaFree(ctx->loop_iters_total);
  mapk::sel_loop_cache_destroy(ctx->loops);
  if (ctx->h_status) cudaFreeHost(ctx->h_status);
  if (ctx->h_done) cudaFreeHost(ctx->h_done);
  if (ctx->s_in) cudaStreamDestroy(ctx->s_in);
  if (ctx->s_out) cudaStreamDestroy(ctx->s_out);
  if (ctx->s_aux) cudaStreamDestroy(ctx->s_aux);
  if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
  if (ctx->ev_join) cudaEventDestroy(ctx->ev_join);
  for (auto& pr : ctx->pairs) { cudaEventDestroy(pr.a); cudaEventDestroy(pr.b); }
  for (auto e : ctx->free_events) cudaEventDestroy(e);
  delete ctx;
}

const char* map_strerror(int code) {
  switch (code) {
    case MAP_OK: return "ok";
    case MAP_EINVAL: return "invalid argument";
    case MAP_ENOMEM: return "out of memory";
    case MAP_ECUDA: return "CUDA error";
    case MAP_ETIMEOUT: return "device-side wait timed out";
    case MAP_EUNSUPPORTED: return "unsupported shape";
    case MAP_EINTERNAL: return "device-side consistency check failed";
    default: return "unknown error";
  }
}

int map_get_counters(map_ctx* ctx, map_counters* out) {
  if (!ctx || !out) return MAP_EINVAL;
  *out = ctx->counters;
  long long iters = 0;   // iterations of the device-side selection loop (completed work)
  if (cudaSetDevice(ctx->device) != cudaSuccess ||
      cudaMemcpy(&iters, ctx->loop_iters_total, sizeof(iters), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MAP_ECUDA;
  out->launches += mapk::kSelLoopKernelsPerIter * iters;
  out->select_rounds += iters;
  return MAP_OK;
}

int map_set_wait_limit(map_ctx* ctx, long long ns) {
  if (!ctx) return MAP_EINVAL;
  ctx->wait_ns = ns > 0 ? ns : 0;
  return MAP_OK;
}

int map_set_timing(map_ctx* ctx, int enable) {
  if (!ctx) return MAP_EINVAL;
  ctx->timing = enable != 0;
  return MAP_OK;
}

int map_read_timing(map_ctx* ctx, int id, double* total_ms, long long* count) {
  if (!ctx || id < 0 || id >= MAP_K_NUM || !total_ms || !count) return MAP_EINVAL;
  if (cudaDeviceSynchronize() != cudaSuccess) return MAP_ECUDA;
  for (auto& pr : ctx->pairs) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, pr.a, pr.b);
    ctx->t_ms[pr.id] += ms;
    ctx->t_n[pr.id] += 1;
    ctx->free_events.push_back(pr.a);
    ctx->free_events.push_back(pr.b);
  }
  ctx->pairs.clear();
  *total_ms = ctx->t_ms[id];
  *count = ctx->t_n[id];
  ctx->t_ms[id] = 0;
  ctx->t_n[id] = 0;
  return MAP_OK;
}

int map_linear(map_ctx* ctx, const void* x, const void* w, const void* b, int M, int K, int Nout, int epi, void* y,
               void* stream) {
  if (!ctx || !x || !w || !y || M < 0 || K <= 0 || Nout <= 0) return MAP_EINVAL;
  if (epi != mapk::EPI_GELU_BF16 && epi != mapk::EPI_BIAS_BF16 && epi != mapk::EPI_F32) return MAP_EINVAL;
  if (K % 64 != 0 || Nout % 64 != 0) return MAP_EUNSUPPORTED;
  if (!aligned16(x) || !aligned16(w) || !aligned16(y)) return MAP_EINVAL;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return MAP_ECUDA;
  GemmDesc d = linear_desc(ctx, x, M, K, w, Nout, epi == mapk::EPI_F32 ? nullptr : b, y, epi);
  return gemm(ctx, d, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
