// Persistent tcgen05 GEMM for sm_103a:  C = epilogue(A @ B^T), A [M, K], B [N, K] bf16.
//
// Used for every dense contraction of the pruning path: the predictor layers f_V, f_T
// (Linear -> GELU -> Linear), the W_K / W_Q projections with RoPE fused into the
// epilogue (section "Cross-Modal Attention Distillation"), Eq. 3's logits, the projection of
// every token on the R0 basis (Eq. 4), and the distillation step.
//
// Structure (one CTA per SM, 6 warps):
//   warp 0      one thread issues TMA loads of 128x64 (A) and BNx64 (B) bf16 tiles, 128-byte
//               swizzled, into a STAGES-deep shared-memory ring (mbarrier full/empty).
//   warp 1      allocates TMEM (2 accumulators x BN fp32 columns); one thread issues
//               tcgen05.mma (M=128, N=BN, K=16) x 4 per stage and commits to mbarriers.
//   CG2 (the BN = 256 predictor layers): 2-CTA clusters run 2-SM MMAs (cta_group::2,
//               M = 256): each CTA loads its 128 A rows and half of the B tile, both
//               complete on the leader's full barrier, the leader's thread issues the MMAs and
//               its commits release the stage and the accumulator in both CTAs.
//   warps 2-5   epilogue: tcgen05.ld the accumulator (one TMEM lane = one output row per
//               thread), apply bias / GELU / RoPE, store (bf16, bf16 hi/lo pair, or fp32);
//               release the accumulator so the
//               MMA warp can start the tile after next while this one drains.
//   EPI_PROJECT: the MMA thread also accumulates A A^T (N = 128) of every stage into a second
//               TMEM accumulator, whose diagonal is ||row||^2.  K is taken in kGramSlices slices,
//               an accumulator each (two, alternating).  Warps 6-9 add them in slice order, the Gram
//               kernel's, in registers and hand a tile's sums to the epilogue warps in a third TMEM
//               region, so that the substitution of one tile runs beside the products of the next.
//               (With the additions in the epilogue warps themselves the MMAs waited for the
//               substitution: calls on 64 images of 2880 tokens took 6 % longer than with one
//               accumulation over K, this way 0.7 %, on one image 2 %.)
// All waits are bounded (ptx.cuh); a timeout sets ST_TIMEOUT and every role drains and exits.
#include <algorithm>
#include <cstdio>
#include <cudaTypedefs.h>

#include "kernels.h"
#include "ptx.cuh"

namespace mapk {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;

// What the two row groups of one launch do not share (GemmDesc's fields of the same names).
struct RowGroup {
  int M;
  void* C;
  const __nv_bfloat16* bias;
  const float* biasf;
  const int* pos; int pos_mod;
  int split_kind; float scale; float* aux;
  const int* seg_valid; int seg_len;
};

struct KArgs {
  RowGroup grp[2]; int groups;
  int M, N, K, batch, a_row_stride, b_row_stride;
  const int* n_limit;
  long long ldc; long long c_batch_stride;
  const float2* rope; int rope_half; int rope_ld;
  int* status;
  const int* b_off;
  float2* stats; int stat_ld; int stat_parts;
  const int* col_count;
  int b_base;
  ProjArgs proj;
  int a_kwrap;
  int split3;
  const int* blist; const int* bcount;
  const int* m_limit;
  unsigned long long wait_ns;   // limit of the role waits (the drain waits keep kWaitLimitNs)
  int ksplit; long long c_split_stride;   // EPI_F32 split-K: partial sums per K slice
  int box_store;                           // EPI_F32: C written by box stores
  GemmProducts pr;                         // EPI_F32: products of column segments (pr.n > 0)
};

__device__ __forceinline__ float gelu_erf(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);   // .x = a (low half), .y = b
  return *reinterpret_cast<uint32_t*>(&h);
}

constexpr int kProjMaxBasis = 128;             // EPI_PROJECT: R0 basis size supported

template <int BN, int STAGES, int EPI, bool CG2>
struct Smem {
  static constexpr bool PROJ = EPI == EPI_PROJECT;
  static constexpr uint32_t A_BYTES = kBM * kBK * 2;
  static constexpr uint32_t B_BYTES = (CG2 ? BN / 2 : BN) * kBK * 2;   // CG2: this CTA's half
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t TILES = STAGES * STAGE_BYTES;
  static constexpr bool EGSYNC = PROJ || EPI == EPI_SM_MEAN;   // epilogue warps' group barrier
  // PROJ: also dempty, sfull and sempty, and one unused: L, which follows, is read 16 bytes at a time
  static constexpr uint32_t XBARS = (EGSYNC ? 1 : 0) + (PROJ ? 4 : 0);
  static constexpr uint32_t BARS = (2 * STAGES + 5 + XBARS) * 8;
  // per-warp 32x32 transposes (EPI_SM_STATS) or the tile's column normalisers (EPI_SM_MEAN)
  static constexpr uint32_t XPOSE = EPI == EPI_SM_STATS ? 4 * 32 * 33 * 4 : (EPI == EPI_SM_MEAN ? BN * 4 : 0);
  // bf16 outputs written by TMA box stores from per-warp staging: hi/lo split epilogues use two
  // buffers of (hi, lo) 32x32 boxes, EPI_ROPE_SPLIT3 (BN = 128) one buffer of (hi, lo) x 2 halves
  static constexpr bool TSTORE_ROPE = EPI == EPI_ROPE_SPLIT3 && BN == 128;
  static constexpr bool TSTORE = EPI == EPI_GELU_SPLIT || EPI == EPI_BIAS_SPLIT || TSTORE_ROPE;
  // EPI_F32: two 32x32 fp32 boxes a warp
  static constexpr bool TSTORE_F32 = EPI == EPI_F32;
  static constexpr uint32_t STG = TSTORE || TSTORE_F32 ? 4 * 4 * 32 * 32 * 2 : 0;
  static constexpr uint32_t LSM = PROJ ? BN * BN * 4 : 0;       // L rows of the basis (pitch BN)
  static constexpr uint32_t PEXTRA = PROJ ? (BN + kBM) * 4 : 0;  // 1/r of the basis, ||row||^2 of the tile
  static constexpr uint32_t TOTAL = 1024 + TILES + STG + BARS + 16 + XPOSE + LSM + PEXTRA;
  static constexpr uint32_t TMEM_COLS =                           // a power of two; PROJ: + the sums, A A^T
      PROJ ? (3 * BN + kBM <= 256 ? 256u : 512u) : (2 * BN > 256 ? 512u : 2 * BN);
  static constexpr int THREADS = PROJ ? 320 : 192;
  static_assert(!PROJ || (TILES + STG + BARS + 16 + XPOSE) % 16 == 0, "float4 reads of L");
};

// Selection value, squared: p^2 * rho^(2 lambda) orders candidates like p * rho^lambda (both are
// >= 0) and needs no square root for lambda = 1.  rho^2 = r2 unless r2 <= tau ||v||^2 (then 0).
__device__ __forceinline__ float proj_value(float p, float r2, float sq, float lam, float tau) {
  if (!(p > 0.f)) return 0.f;
  if (lam == 0.f) return p * p;
  if (!(r2 > tau * sq) || !(r2 > 0.f)) return 0.f;
  const float v = lam == 1.f ? (p * p) * r2 : (p * p) * powf(r2, lam);
  return v > 0.f ? v : 0.f;
}

struct TileCoord { int b, m_blk, n_blk, ks, grp; bool skip; };

// The tensor maps of a launch: A, B and the box-stored output of each row group.
struct Maps { CUtensorMap A[2], B[2], C[2]; };

// Work unit t -> tile.  With PAIR the unit is a pair of vertically adjacent M tiles with the
// same N tile, processed by the two CTAs of a cluster (rank 0 the upper, rank 1 the lower).
// With split-K (ksplit > 1) a unit is also one K slice ks of its tile.
// PROJECT (one column tile, no split-K) with m_limit: only the row tiles with rows of an image are
// units, found by a walk over the listed images (up to 64; with more, tiles past an image's rows are
// skipped where they come up).
constexpr int kProjWalkMax = 64;
__device__ inline bool proj_walks(const KArgs& a, int nbatch) { return a.m_limit && nbatch <= kProjWalkMax; }
// Image (list position) and row tile of unit t, or, when t is past the units, b = -1 - (their number).
__device__ inline void proj_walk(const KArgs& a, int nbatch, int t, int& b, int& mu) {
  int found = 0;
  for (int i = 0; i < nbatch; ++i) {
    const int img = a.blist ? __ldg(a.blist + i) : i;
    const int n = (min(a.M, __ldg(a.m_limit + img)) + kBM - 1) / kBM;
    if (t < found + n) {
      b = i;
      mu = t - found;
      return;
    }
    found += n;
  }
  b = -1 - found;
  mu = 0;
}

template <bool PAIR, bool PROJECT>
__device__ __forceinline__ TileCoord tile_coord(const KArgs& a, int t, int nbatch, int m_units, int n_tiles, int BN,
                                                uint32_t crank) {
  TileCoord c;
  int mu;
  if (PROJECT && proj_walks(a, nbatch)) {
    proj_walk(a, nbatch, t, c.b, mu);
    c.ks = c.n_blk = 0;
  } else {
    const int tiles = m_units * n_tiles;
    const int per = tiles * a.ksplit;
    c.b = t / per;
    int rem = t - c.b * per;
    c.ks = rem / tiles;
    rem -= c.ks * tiles;
    mu = rem / n_tiles;
    c.n_blk = rem - mu * n_tiles;
  }
  if (a.blist) c.b = __ldg(a.blist + c.b);
  c.m_blk = PAIR ? 2 * mu + static_cast<int>(crank) : mu;
  c.grp = 0;
  int lim = a.n_limit ? min(a.N, __ldg(a.n_limit + c.b)) : a.N;
  c.skip = c.n_blk * BN >= lim;
  if (PROJECT && a.m_limit && mu * kBM >= __ldg(a.m_limit + c.b)) c.skip = true;
  return c;
}

// Row groups: the predictor's two modalities in one launch (same N and K, other rows and weights),
// the units of the first followed by those of the second, so that neither waits for the other's
// last wave.  With seg_valid, a group's rows come in segments of seg_len of which the first
// seg_valid[s] hold data: only row tiles with such rows are units, counted and found by a walk over
// the segments (up to kWalkMax of them: a few hundred cycles a tile; with more, tiles without data
// are skipped where they come up).
constexpr int kWalkMax = 64;

__device__ __forceinline__ bool walks(const RowGroup& q) {
  return q.seg_valid && (q.M + q.seg_len - 1) / q.seg_len <= kWalkMax;
}
// The i-th row tile (of `rows` rows) with data, or, when i is past them, -1 - (their number).
__device__ inline int walk_tiles(const RowGroup& q, int rows, int i) {
  int next = 0, found = 0;                           // first tile not yet counted, tiles counted
  for (int s = 0; s * q.seg_len < q.M; ++s) {
    const int r0 = s * q.seg_len, r1 = min(q.M, r0 + __ldg(q.seg_valid + s));
    const int first = max(r0 / rows, next), last = (r1 - 1) / rows;
    if (r1 <= r0 || last < first) continue;
    if (i < found + last - first + 1) return first + (i - found);
    found += last - first + 1;
    next = last + 1;
  }
  return -1 - found;
}
__device__ __forceinline__ int group_units(const RowGroup& q, int rows) {
  return walks(q) ? -1 - walk_tiles(q, rows, 0x7FFFFFFF) : (q.M + rows - 1) / rows;
}

template <bool PAIR>
__device__ __forceinline__ TileCoord group_coord(const KArgs& a, int t, int units0, int n_tiles, uint32_t crank) {
  constexpr int ROWS = PAIR ? 2 * kBM : kBM;
  TileCoord c;
  c.b = c.ks = 0;
  c.grp = t >= units0 * n_tiles;
  if (c.grp) t -= units0 * n_tiles;
  const RowGroup& q = a.grp[c.grp];
  int mu = t / n_tiles;
  c.n_blk = t - mu * n_tiles;
  c.skip = false;
  if (walks(q)) {
    mu = walk_tiles(q, ROWS, mu);
  } else if (q.seg_valid) {
    const int r0 = mu * ROWS, r1 = min(q.M, r0 + ROWS);
    c.skip = true;
    for (int s = r0 / q.seg_len; s * q.seg_len < r1; ++s)
      if (max(r0, s * q.seg_len) < s * q.seg_len + __ldg(q.seg_valid + s)) c.skip = false;
  }
  c.m_blk = PAIR ? 2 * mu + static_cast<int>(crank) : mu;
  return c;
}

template <int BN, int STAGES, int EPI, bool CG2>
__global__ void __launch_bounds__(Smem<BN, STAGES, EPI, CG2>::THREADS, 1)
gemm_tc_kernel(const __grid_constant__ Maps maps, const __grid_constant__ KArgs a) {
  constexpr bool GROUPED = EPI == EPI_GELU_SPLIT || EPI == EPI_ROPE_SPLIT3;
  using S = Smem<BN, STAGES, EPI, CG2>;
  constexpr bool PAIR = CG2;
  constexpr uint32_t IDESC = idesc_bf16(CG2 ? 2 * kBM : kBM, BN);
  const uint32_t crank = PAIR ? cluster_ctarank() : 0u;
  const int unit0 = PAIR ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int units_step = PAIR ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * S::A_BYTES;
  uint8_t* stg = smem + S::TILES;                // TSTORE staging boxes (1024-aligned)
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::TILES + S::STG);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1 + S::XBARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint64_t* egsync = drain + 1;                  // EGSYNC: epilogue warps' group barrier
  uint64_t* dempty = drain + 2;                  // PROJ: A A^T has been read; the tile's sums are written; read
  uint64_t* sfull = drain + 3;
  uint64_t* sempty = drain + 4;
  float* xpose = reinterpret_cast<float*>(smem + S::TILES + S::STG + S::BARS + 16);
  float* Lsm = xpose + S::XPOSE / 4;
  float* rinv_sm = Lsm + S::LSM / 4;
  float* sq_sm = rinv_sm + BN;                   // PROJ

  // uniform in the warp, and known to be
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    // tempty: one arrive per epilogue warp (of both CTAs with CG2, on the leader's barrier)
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], CG2 ? 8 : 4); }
    mbar_init(drain, 1);
    if constexpr (S::EGSYNC) {
      mbar_init(egsync, 128);
    }
    if constexpr (S::PROJ) {                       // an arrive per warp
      mbar_init(dempty, 4);
      mbar_init(sfull, 4);
      mbar_init(sempty, 4);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&maps.A[0]); tma_prefetch_desc(&maps.B[0]); }
  pdl_enter();                                    // inputs below come from the previous kernel
  if (warp == 1) {
    if constexpr (CG2) { tmem_alloc_cg2(tmem_slot, S::TMEM_COLS); tmem_relinquish_cg2(); }
    else { tmem_alloc(tmem_slot, S::TMEM_COLS); tmem_relinquish(); }
  }
  if constexpr (PAIR) cluster_sync();             // peer barriers initialised before any remote arrive
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int m_tiles = (a.M + kBM - 1) / kBM;
  constexpr int UNIT_ROWS = PAIR ? 2 * kBM : kBM;
  int group0 = 0;                                 // row units of the first group
  if constexpr (GROUPED) group0 = group_units(a.grp[0], UNIT_ROWS);
  const int m_units = PAIR ? (m_tiles + 1) / 2 : m_tiles;
  const int n_tiles = (a.N + BN - 1) / BN;
  const int nbatch = a.blist ? min(a.batch, *a.bcount) : a.batch;
  int total = nbatch * m_units * n_tiles * a.ksplit;
  if constexpr (GROUPED) {
    total = group0;
    if (a.groups > 1) total += group_units(a.grp[1], UNIT_ROWS);
    total *= n_tiles;
  }
  if constexpr (EPI == EPI_PROJECT) {
    if (proj_walks(a, nbatch)) {
      int none;
      proj_walk(a, nbatch, 0x7FFFFFFF, total, none);
      total = -1 - total;
    }
  }
  auto coord = [&](int t) {
    if constexpr (GROUPED) return group_coord<PAIR>(a, t, group0, n_tiles, crank);
    else return tile_coord<PAIR, EPI == EPI_PROJECT>(a, t, nbatch, m_units, n_tiles, BN, crank);
  };
  constexpr bool PRODUCTS = EPI == EPI_F32;       // the epilogue of the segmented products
  constexpr int SLICES = S::PROJ ? kGramSlices : 1;   // accumulators per tile, one after the other
  // K blocks of one product of image c.b
  auto product_kblocks = [&](const TileCoord& c) {
    return a.pr.k_count ? (__ldg(a.pr.k_count + c.b) + kBK - 1) / kBK : a.pr.kblocks;
  };
  // K blocks of a unit's slice (the whole K without split-K)
  auto kb_range = [&](const TileCoord& c, int& kb0, int& kb1) {
    int KB = a.K / kBK;
    if constexpr (PRODUCTS) {
      if (a.pr.n > 0) KB = a.pr.n * product_kblocks(c);
    }
    kb0 = c.ks * KB / a.ksplit;
    kb1 = (c.ks + 1) * KB / a.ksplit;
  };
  // K block kb -> (A column, B column)
  auto kcols = [&](int kb, int& ac, int& bc) {
    if (a.split3) {
      const int nbk = a.K / kBK / 3;
      if (kb < 2 * nbk) {
        const int j = kb >> 1;
        ac = j * kBK;
        bc = (kb & 1) ? (2 * nbk + j) * kBK : j * kBK;
      } else {
        ac = bc = (kb - nbk) * kBK;
      }
    } else {
      ac = a.a_kwrap > 0 ? (kb * kBK) % a.a_kwrap : kb * kBK;
      bc = kb * kBK;
    }
  };

  // Producer: parity of the last load issued into each stage (-1: none), for the drain below.
  int last_par[STAGES];
#pragma unroll
  for (int s = 0; s < STAGES; ++s) last_par[s] = -1;
  bool drains = false;                            // this thread issued the loads
  if (warp == 0) {
    if (elect_one()) {
      // ---------------------------------------------------------------- TMA producer
      drains = true;
      uint32_t stage = 0, phase = 0;
      bool ok = true;
      for (int t = unit0; t < total && ok; t += units_step) {
        TileCoord c = coord(t);
        if (c.skip) continue;
        const int arow = c.b * a.a_row_stride + c.m_blk * kBM;
        const int brow = (a.b_off ? __ldg(a.b_off + c.b) : c.b * a.b_row_stride + a.b_base) + c.n_blk * BN;
        int kb0, kb1;
        kb_range(c, kb0, kb1);
        if constexpr (PRODUCTS) {
          if (a.pr.n > 0) {
            // K block k0 of product p: segment p of each operand, K-major (one box of rows) or
            // MN-major (boxes of 64 columns by 64 K rows: the operand's rows are its K index).  One
            // thread issues every load, so what a K block does not change is kept out of its loop.
            const GemmProducts& q = a.pr;
            constexpr int BR = CG2 ? BN / 2 : BN;
            const int nkb = product_kblocks(c);
            const int n0 = c.n_blk * BN + (CG2 ? static_cast<int>(crank) * BR : 0), m0 = c.m_blk * kBM;
            const int arb = q.a_off ? __ldg(q.a_off + c.b) : c.b * a.a_row_stride;
            const int brb = q.b_off ? __ldg(q.b_off + c.b) : c.b * a.b_row_stride;
            const bool amn = q.a_mn != 0, bmn = q.b_mn != 0;
            int p = kb0 / nkb, j = kb0 - p * nkb;
            int aseg = q.a_seg[p], bseg = q.b_seg[p];
            const uint32_t fb0 = CG2 ? mapa_u32(full, 0) : 0u;
            for (int kb = kb0; kb < kb1; ++kb) {
              if (!mbar_wait(&empty[stage], phase ^ 1, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
              const uint32_t fb = fb0 + stage * 8;
              if constexpr (CG2) {
                if (crank == 0) mbar_arrive_expect_tx(&full[stage], 2 * S::STAGE_BYTES);
              } else {
                mbar_arrive_expect_tx(&full[stage], S::STAGE_BYTES);
              }
              auto load = [&](uint8_t* dst, const CUtensorMap* tm, int x, int y) {
                if constexpr (CG2) tma_load_2d_cg2(dst, tm, fb, x, y);
                else tma_load_2d(dst, tm, &full[stage], x, y);
              };
              uint8_t* da = sA + stage * S::A_BYTES;
              uint8_t* db = sB + stage * S::B_BYTES;
              const int k0 = j * kBK;
              if (amn) {
#pragma unroll
                for (int h = 0; h < kBM; h += 64) load(da + h * 128, &maps.A[0], aseg + m0 + h, arb + k0);
              } else {
                load(da, &maps.A[0], aseg + k0, arb + m0);
              }
              if (bmn) {
#pragma unroll
                for (int h = 0; h < BR; h += 64) load(db + h * 128, &maps.B[0], bseg + n0 + h, brb + k0);
              } else {
                load(db, &maps.B[0], bseg + k0, brb + n0);
              }
              last_par[stage] = static_cast<int>(phase);
              if (++stage == STAGES) { stage = 0; phase ^= 1; }
              if (++j == nkb && kb + 1 < kb1) {
                j = 0;
                ++p;
                aseg = q.a_seg[p];
                bseg = q.b_seg[p];
              }
            }
            continue;
          }
        }
        const CUtensorMap* const tmA = &maps.A[GROUPED ? c.grp : 0];
        const CUtensorMap* const tmB = &maps.B[GROUPED ? c.grp : 0];
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(&empty[stage], phase ^ 1, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
          int ac, bc;
          kcols(kb, ac, bc);
          if constexpr (CG2) {
            // both CTAs' copies complete on the leader's full barrier, which expects them all
            if (crank == 0) mbar_arrive_expect_tx(&full[stage], 2 * S::STAGE_BYTES);
            const uint32_t fb = mapa_u32(&full[stage], 0);
            tma_load_2d_cg2(sA + stage * S::A_BYTES, tmA, fb, ac, arow);
            tma_load_2d_cg2(sB + stage * S::B_BYTES, tmB, fb, bc, brow + static_cast<int>(crank) * (BN / 2));
          } else {
            mbar_arrive_expect_tx(&full[stage], S::STAGE_BYTES);
            tma_load_2d(sA + stage * S::A_BYTES, tmA, &full[stage], ac, arow);
            tma_load_2d(sB + stage * S::B_BYTES, tmB, &full[stage], bc, brow);
          }
          last_par[stage] = static_cast<int>(phase);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (crank == 0 && elect_one()) {
      // ---------------------------------------------------------------- MMA issuer (CG2: leader)
      uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
      [[maybe_unused]] uint32_t d_phase = 0;
      bool issued = false, ok = true;
      // descriptors without their address (shared memory addresses are below 2^18); products: also
      // their step per 16 K: 32 bytes along a K-major row, 16 rows of 128 bytes of an MN-major box
      const uint64_t kdesc0 = desc_sw128(0);
      const bool amn = PRODUCTS && a.pr.a_mn, bmn = PRODUCTS && a.pr.b_mn;
      const uint64_t adesc0 = amn ? desc_sw128_mn(0) : desc_sw128(0), bdesc0 = bmn ? desc_sw128_mn(0) : desc_sw128(0);
      const uint32_t astep = (amn ? 2048 : 32) >> 4, bstep = (bmn ? 2048 : 32) >> 4;
      const uint32_t pid = IDESC | (amn ? 1u << 15 : 0u) | (bmn ? 1u << 16 : 0u);
      for (int t = unit0; t < total && ok; t += units_step) {
        TileCoord c = coord(t);
        if (c.skip) continue;
        for (int sl = 0; sl < SLICES; ++sl) {
          int kb0, kb1;
          kb_range(c, kb0, kb1);
          if constexpr (S::PROJ) {
            kb0 = sl * (a.K / kBK) / kGramSlices;
            kb1 = (sl + 1) * (a.K / kBK) / kGramSlices;
            if (kb0 == kb1) continue;                // fewer K blocks than slices
          }
          if (!mbar_wait(&tempty[acc], acc_phase ^ 1, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * BN;
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait(&full[stage], phase, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA + stage * S::A_BYTES);
            const uint32_t b0 = smem_u32(sB + stage * S::B_BYTES);
            if (PRODUCTS && a.pr.n > 0) {
#pragma unroll
              for (int k = 0; k < kBK / 16; ++k) {
                const uint64_t da = adesc0 + (a0 >> 4) + k * astep, db = bdesc0 + (b0 >> 4) + k * bstep;
                if constexpr (CG2) umma_bf16_cg2(d_tmem, da, db, pid, (kb != kb0 || k != 0));
                else umma_bf16(d_tmem, da, db, pid, (kb != kb0 || k != 0));
              }
              if constexpr (CG2) umma_commit_cg2_mc(&empty[stage], static_cast<uint16_t>(3));
              else umma_commit(&empty[stage]);
            } else if constexpr (CG2) {
              const uint64_t da = kdesc0 + (a0 >> 4), db = kdesc0 + (b0 >> 4);
#pragma unroll
              for (int k = 0; k < kBK / 16; ++k) umma_bf16_cg2(d_tmem, da + 2 * k, db + 2 * k, IDESC, (kb != kb0 || k != 0));
              umma_commit_cg2_mc(&empty[stage], static_cast<uint16_t>(3));
            } else {
              const uint64_t da = kdesc0 + (a0 >> 4), db = kdesc0 + (b0 >> 4);
#pragma unroll
              for (int k = 0; k < kBK / 16; ++k) umma_bf16(d_tmem, da + 2 * k, db + 2 * k, IDESC, (kb != kb0 || k != 0));
              issued = true;
              if constexpr (S::PROJ) {   // A A^T: its diagonal is ||row||^2
                if (kb == kb0) {         // the previous slice's has been read
                  if (!mbar_wait(dempty, d_phase ^ 1, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
                  tc_fence_after();
                  d_phase ^= 1;
                }
                const uint32_t n_tmem = tmem_base + 3 * BN;
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k)
                  umma_bf16(n_tmem, da + 2 * k, da + 2 * k, idesc_bf16(kBM, kBM), (kb != kb0 || k != 0));
              }
              umma_commit(&empty[stage]);
            }
            issued = true;
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
          if (!ok) break;
          if constexpr (CG2) umma_commit_cg2_mc(&tfull[acc], static_cast<uint16_t>(3));
          else umma_commit(&tfull[acc]);
          acc ^= 1;
          if (acc == 0) acc_phase ^= 1;
        }
      }
      if (issued) {   // every MMA of this CTA has completed before TMEM is released
        if constexpr (CG2) umma_commit_cg2(drain);
        else umma_commit(drain);
        mbar_wait(drain, 0, a.status, nullptr);
      }
    }
    __syncwarp();
  } else if (warp < 6) {
    // ------------------------------------------------------------------ epilogue
    const int lane_grp = warp & 3;                 // TMEM lanes this warp may access
    const int r_in_tile = lane_grp * 32 + lane;
    uint32_t acc = 0, acc_phase = 0;
    int staged_b = -1;                             // EPI_PROJECT: image whose L is in shared memory
    uint32_t eg_phase = 0;
    bool eg_ok = true;
    for (int t = unit0; t < total && eg_ok; t += units_step) {
      TileCoord c = coord(t);
      if (c.skip) continue;
      if constexpr (S::PROJ) {
        if (c.b != staged_b) {                     // stage L and 1/r of this image's R0 basis
          // group barrier of the 128 epilogue threads (bounded, unlike a named barrier)
          mbar_arrive(egsync);
          if (!mbar_wait(egsync, eg_phase, a.status, abort_flag, a.wait_ns)) { eg_ok = false; break; }
          eg_phase ^= 1;
          const ProjArgs& pj = a.proj;
          const int nb0 = min(BN, __ldg(pj.nbasis + c.b));
          const long long ibase = static_cast<long long>(c.b) * a.M;
          const int KV = BN / 4;
          for (int t4 = threadIdx.x - 64; t4 < nb0 * KV; t4 += 128) {
            const int i = t4 / KV, q = (t4 - i * KV) * 4;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q < i) {
              const int tk = __ldg(pj.basis_tok + static_cast<long long>(c.b) * pj.Kcap + i);
              const float* row = pj.Ec + (ibase + tk) * pj.KP + q;
              v.x = row[0];
              v.y = q + 1 < i ? row[1] : 0.f;
              v.z = q + 2 < i ? row[2] : 0.f;
              v.w = q + 3 < i ? row[3] : 0.f;
            }
            *reinterpret_cast<float4*>(Lsm + i * BN + q) = v;
          }
          for (int i = threadIdx.x - 64; i < nb0; i += 128)
            rinv_sm[i] = 1.0f / __ldg(pj.rnorm + static_cast<long long>(c.b) * pj.Kcap + i);
          mbar_arrive(egsync);
          if (!mbar_wait(egsync, eg_phase, a.status, abort_flag, a.wait_ns)) { eg_ok = false; break; }
          eg_phase ^= 1;
          staged_b = c.b;
        }
      }
      if constexpr (EPI == EPI_SM_MEAN) {
        // the tile's column normalisers c = max + ln(sum), +inf past the image's columns (exp(-inf) =
        // 0): read, or, when stat_parts is given, combined here from the slabs' partial (max, sum) while the
        // MMAs run, in stats_combine_kernel's order (eight interleaved sums, then their sum)
        mbar_arrive(egsync);                       // the previous tile's are no longer read
        if (!mbar_wait(egsync, eg_phase, a.status, abort_flag, a.wait_ns)) { eg_ok = false; break; }
        eg_phase ^= 1;
        const int ncols = min(a.n_limit ? min(a.N, __ldg(a.n_limit + c.b)) : a.N,
                              a.col_count ? __ldg(a.col_count + c.b) : a.N);
        for (int j = threadIdx.x - 64; j < BN; j += 128) {
          const int col = c.n_blk * BN + j;
          float v = INFINITY;
          if (col < ncols) {
            if (a.stat_parts > 0) {
              const float2* p = a.stats + static_cast<long long>(c.b) * a.stat_parts * a.stat_ld + col;
              float m = -INFINITY;
#pragma unroll 8
              for (int i = 0; i < a.stat_parts; ++i) m = fmaxf(m, p[static_cast<long long>(i) * a.stat_ld].x);
              float s8[8];
#pragma unroll
              for (int y = 0; y < 8; ++y) s8[y] = 0.f;
              for (int i0 = 0; i0 < a.stat_parts; i0 += 8) {
                float2 w[8];
#pragma unroll
                for (int y = 0; y < 8; ++y)
                  w[y] = i0 + y < a.stat_parts ? p[static_cast<long long>(i0 + y) * a.stat_ld] : make_float2(0.f, 0.f);
#pragma unroll
                for (int y = 0; y < 8; ++y)
                  if (w[y].y > 0.f) s8[y] += w[y].y * expf(w[y].x - m);
              }
              float s = s8[0];
#pragma unroll
              for (int y = 1; y < 8; ++y) s += s8[y];
              v = m + logf(s);
            } else {
              v = __ldg(a.stats + static_cast<long long>(c.b) * a.stat_ld + col).x;
            }
          }
          xpose[j] = v;
        }
        mbar_arrive(egsync);
        if (!mbar_wait(egsync, eg_phase, a.status, abort_flag, a.wait_ns)) { eg_ok = false; break; }
        eg_phase ^= 1;
      }
      const int row = c.m_blk * kBM + r_in_tile;
      const RowGroup& q = a.grp[GROUPED ? c.grp : 0];
      const bool row_ok = row < (a.m_limit ? min(q.M, __ldg(a.m_limit + c.b)) : q.M);
      const int lim = a.n_limit ? min(a.N, __ldg(a.n_limit + c.b)) : a.N;
      const int col0 = c.n_blk * BN;
      // the RoPE factors the epilogue starts with are loaded while the tile's MMAs still run
      [[maybe_unused]] float2 cs[32];
      [[maybe_unused]] const float2* rt = nullptr;
      [[maybe_unused]] auto load_rope = [&](int i0) {
#pragma unroll
        for (int j = 0; j < 32; ++j) cs[j] = __ldg(rt + static_cast<long long>(i0 + j) * a.rope_ld);
      };
      if constexpr (S::TSTORE_ROPE) {
        int pos = 0;
        if (row_ok) pos = q.pos ? __ldg(q.pos + row) : row % q.pos_mod;
        rt = a.rope + pos;
        load_rope(0);
      }
      // EPI_PROJECT: the tile's sums, in their own region
      if (!mbar_wait(S::PROJ ? sfull : &tfull[acc], acc_phase, a.status, abort_flag, a.wait_ns)) break;
      tc_fence_after();
      const uint32_t tbase =
          tmem_base + (static_cast<uint32_t>(lane_grp * 32) << 16) + (S::PROJ ? 2 * BN : acc * BN);
      const long long crow = static_cast<long long>(c.b) * a.c_batch_stride + static_cast<long long>(row) * a.ldc;

      if constexpr (EPI == EPI_ROPE_F32) {
        // BN == dp: the whole row is in this tile; rotate pairs (i, i + dp/2).
        constexpr int HALF = BN / 2;
        float* out = reinterpret_cast<float*>(q.C) + crow;
        int pos = 0;
        if (row_ok) pos = q.pos ? __ldg(q.pos + row) : row % q.pos_mod;
        const float2* rt = a.rope + pos;
#pragma unroll 1
        for (int ch = 0; ch < HALF / 32; ++ch) {
          uint32_t r1[32], r2[32];
          tmem_ld32(tbase + ch * 32, r1);
          tmem_ld32(tbase + HALF + ch * 32, r2);
          if (row_ok) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
              float o1[4], o2[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float2 cs = __ldg(rt + static_cast<long long>(ch * 32 + j + u) * a.rope_ld);
                const float x1 = __uint_as_float(r1[j + u]), x2 = __uint_as_float(r2[j + u]);
                o1[u] = x1 * cs.x - x2 * cs.y;
                o2[u] = x2 * cs.x + x1 * cs.y;
              }
              *reinterpret_cast<float4*>(out + ch * 32 + j) = make_float4(o1[0], o1[1], o1[2], o1[3]);
              *reinterpret_cast<float4*>(out + HALF + ch * 32 + j) = make_float4(o2[0], o2[1], o2[2], o2[3]);
            }
          }
        }
      } else if constexpr (S::TSTORE_ROPE) {
        // BN == dp = 128; x = RoPE(acc + bias) * scale as bf16 (hi, lo) segments, staged per warp
        // in shared memory and written by TMA box stores (rows past M are clipped)
        constexpr int HALF = BN / 2;
        float* aux = (q.aux && row_ok) ? q.aux + static_cast<long long>(row) * BN : nullptr;
        const int seg_lo = q.split_kind == 0 ? 1 : 2;   // keys [hi, lo, hi], queries [hi, hi, lo]
        const int ew = warp - 2;
        const int y = c.b * a.a_row_stride + c.m_blk * kBM + lane_grp * 32;
        uint8_t* sb = stg + ew * 8192;                 // [hi1 | lo1 | hi2 | lo2], 32 rows x 64 B each
#pragma unroll 1
        for (int ch = 0; ch < HALF / 32; ++ch) {
          uint32_t r1[32], r2[32];
          if (ch > 0) load_rope(ch * 32);
          tmem_ld32(tbase + ch * 32, r1);
          tmem_ld32(tbase + HALF + ch * 32, r2);
          if (lane == 0) bulk_wait_group_read<0>();    // the previous chunk's stores have read sb
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 32; j += 8) {
            float o1[8], o2[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const float2 rc = cs[j + u];
              float x1 = __uint_as_float(r1[j + u]), x2 = __uint_as_float(r2[j + u]);
              if (q.biasf) {
                x1 += __ldg(q.biasf + ch * 32 + j + u);
                x2 += __ldg(q.biasf + HALF + ch * 32 + j + u);
              }
              o1[u] = x1 * rc.x - x2 * rc.y;
              o2[u] = x2 * rc.x + x1 * rc.y;
            }
            if (aux) {
#pragma unroll
              for (int u = 0; u < 8; u += 4) {
                *reinterpret_cast<float4*>(aux + ch * 32 + j + u) = make_float4(o1[u], o1[u + 1], o1[u + 2], o1[u + 3]);
                *reinterpret_cast<float4*>(aux + HALF + ch * 32 + j + u) =
                    make_float4(o2[u], o2[u + 1], o2[u + 2], o2[u + 3]);
              }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) { o1[u] *= q.scale; o2[u] *= q.scale; }
            uint32_t h1[4], l1[4], h2[4], l2[4];
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
              const __nv_bfloat162 a1 = __floats2bfloat162_rn(o1[u], o1[u + 1]);
              const __nv_bfloat162 a2 = __floats2bfloat162_rn(o2[u], o2[u + 1]);
              h1[u / 2] = *reinterpret_cast<const uint32_t*>(&a1);
              h2[u / 2] = *reinterpret_cast<const uint32_t*>(&a2);
              l1[u / 2] = pack_bf16(o1[u] - __bfloat162float(a1.x), o1[u + 1] - __bfloat162float(a1.y));
              l2[u / 2] = pack_bf16(o2[u] - __bfloat162float(a2.x), o2[u + 1] - __bfloat162float(a2.y));
            }
            uint8_t* rowp = sb + lane * 64 + ((j / 8) ^ ((lane >> 1) & 3)) * 16;   // 64-byte swizzle
            *reinterpret_cast<uint4*>(rowp) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
            *reinterpret_cast<uint4*>(rowp + 2048) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
            *reinterpret_cast<uint4*>(rowp + 4096) = make_uint4(h2[0], h2[1], h2[2], h2[3]);
            *reinterpret_cast<uint4*>(rowp + 6144) = make_uint4(l2[0], l2[1], l2[2], l2[3]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
#pragma unroll
            for (int sg = 0; sg < 3; ++sg) {
              const int x = sg * BN + ch * 32;
              tma_store_2d(&maps.C[GROUPED ? c.grp : 0], sb + (sg == seg_lo ? 2048 : 0), x, y);
              tma_store_2d(&maps.C[GROUPED ? c.grp : 0], sb + (sg == seg_lo ? 6144 : 4096), x + HALF, y);
            }
            bulk_commit_group();
          }
        }
      } else if constexpr (EPI == EPI_ROPE_SPLIT3) {
        // BN == dp; x = RoPE(acc) * scale, stored as bf16 (hi, lo) segments
        constexpr int HALF = BN / 2;
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(q.C) + crow;
        float* aux = q.aux ? q.aux + static_cast<long long>(row) * BN : nullptr;
        int pos = 0;
        if (row_ok) pos = q.pos ? __ldg(q.pos + row) : row % q.pos_mod;
        const float2* rt = a.rope + pos;
        // segment order: keys [hi, lo, hi], queries [hi, hi, lo]
        const int seg_lo = q.split_kind == 0 ? 1 : 2;
#pragma unroll 1
        for (int ch = 0; ch < HALF / 32; ++ch) {
          uint32_t r1[32], r2[32];
          tmem_ld32(tbase + ch * 32, r1);
          tmem_ld32(tbase + HALF + ch * 32, r2);
          if (row_ok) {
#pragma unroll
            for (int j = 0; j < 32; j += 8) {
              float o1[8], o2[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const float2 cs = __ldg(rt + static_cast<long long>(ch * 32 + j + u) * a.rope_ld);
                float x1 = __uint_as_float(r1[j + u]), x2 = __uint_as_float(r2[j + u]);
                if (q.biasf) {
                  x1 += __ldg(q.biasf + ch * 32 + j + u);
                  x2 += __ldg(q.biasf + HALF + ch * 32 + j + u);
                }
                o1[u] = x1 * cs.x - x2 * cs.y;
                o2[u] = x2 * cs.x + x1 * cs.y;
              }
              if (aux) {
#pragma unroll
                for (int u = 0; u < 8; u += 4) {
                  *reinterpret_cast<float4*>(aux + ch * 32 + j + u) = make_float4(o1[u], o1[u + 1], o1[u + 2], o1[u + 3]);
                  *reinterpret_cast<float4*>(aux + HALF + ch * 32 + j + u) =
                      make_float4(o2[u], o2[u + 1], o2[u + 2], o2[u + 3]);
                }
              }
#pragma unroll
              for (int u = 0; u < 8; ++u) { o1[u] *= q.scale; o2[u] *= q.scale; }
              uint32_t h1[4], l1[4], h2[4], l2[4];
#pragma unroll
              for (int u = 0; u < 8; u += 2) {
                const __nv_bfloat162 a1 = __floats2bfloat162_rn(o1[u], o1[u + 1]);
                const __nv_bfloat162 a2 = __floats2bfloat162_rn(o2[u], o2[u + 1]);
                h1[u / 2] = *reinterpret_cast<const uint32_t*>(&a1);
                h2[u / 2] = *reinterpret_cast<const uint32_t*>(&a2);
                l1[u / 2] = pack_bf16(o1[u] - __bfloat162float(a1.x), o1[u + 1] - __bfloat162float(a1.y));
                l2[u / 2] = pack_bf16(o2[u] - __bfloat162float(a2.x), o2[u + 1] - __bfloat162float(a2.y));
              }
              const uint4 H1 = make_uint4(h1[0], h1[1], h1[2], h1[3]), L1 = make_uint4(l1[0], l1[1], l1[2], l1[3]);
              const uint4 H2 = make_uint4(h2[0], h2[1], h2[2], h2[3]), L2 = make_uint4(l2[0], l2[1], l2[2], l2[3]);
#pragma unroll
              for (int sg = 0; sg < 3; ++sg) {
                __nv_bfloat16* o = out + sg * BN + ch * 32 + j;
                *reinterpret_cast<uint4*>(o) = sg == seg_lo ? L1 : H1;
                *reinterpret_cast<uint4*>(o + HALF) = sg == seg_lo ? L2 : H2;
              }
            }
          }
        }
      } else if constexpr (EPI == EPI_SM_STATS) {
        // column max / sum of exp over this warp's 32 rows (rows past M count as -inf):
        // the 32x32 chunk is transposed through shared memory, lane j reduces column j.
        float2* part = a.stats + (static_cast<long long>(c.b) * m_tiles * 4 + c.m_blk * 4 + lane_grp) * a.stat_ld;
        const int ncol = a.col_count ? min(lim, __ldg(a.col_count + c.b)) : lim;
        float* tr = xpose + (warp - 2) * 32 * 33;
#pragma unroll 1
        for (int ch = 0; ch < BN / 32; ++ch) {
          uint32_t r[32];
          tmem_ld32(tbase + ch * 32, r);
          const int cbase = col0 + ch * 32;
          if (cbase >= ncol) continue;                    // uniform in the warp
#pragma unroll
          for (int j = 0; j < 32; ++j) tr[lane * 33 + j] = row_ok ? __uint_as_float(r[j]) : -INFINITY;
          __syncwarp();
          float m = -INFINITY;
#pragma unroll
          for (int i = 0; i < 32; ++i) m = fmaxf(m, tr[i * 33 + lane]);
          float sum = 0.f;
          if (m != -INFINITY) {
#pragma unroll
            for (int i = 0; i < 32; ++i) sum += __expf(tr[i * 33 + lane] - m);
          }
          __syncwarp();
          if (cbase + lane < ncol) part[cbase + lane] = make_float2(m, sum);
        }
      } else if constexpr (EPI == EPI_SM_MEAN) {
        // p_hat[row] = (1/M_b) sum_col exp(l - c_col), the c_col read as broadcasts
        const int ncol = a.col_count ? min(lim, __ldg(a.col_count + c.b)) : lim;
        float acc_p = 0.f;
#pragma unroll 1
        for (int ch = 0; ch < BN / 32; ++ch) {
          uint32_t r[32];
          tmem_ld32(tbase + ch * 32, r);
          if (col0 + ch * 32 >= ncol) continue;           // uniform in the warp
          const float* cn = xpose + ch * 32;
#pragma unroll
          for (int j = 0; j < 32; ++j) acc_p += __expf(__uint_as_float(r[j]) - cn[j]);
        }
        if (row < a.M) {   // rows past the image's valid tokens (m_limit) get 0
          float* out = reinterpret_cast<float*>(q.C) + static_cast<long long>(c.b) * a.c_batch_stride;
          out[static_cast<long long>(c.n_blk) * a.M + row] =
              row_ok ? acc_p / static_cast<float>(ncol > 0 ? ncol : 1) : 0.f;
        }
      } else if constexpr (EPI == EPI_PROJECT) {
        // Cholesky coordinates of token `row` on the R0 basis by forward substitution,
        // 32 basis vectors at a time: e_beta = (g_beta - sum_{q<beta} L[beta][q] e_q) / r_beta.
        // Each finished chunk of e replaces its g columns in TMEM, where later chunks read it.
        const ProjArgs& pj = a.proj;
        const int nb0 = min(BN, __ldg(pj.nbasis + c.b));
        const long long tok = static_cast<long long>(c.b) * a.M + row;
        const bool alive = row_ok && __ldg(pj.state + tok) == 0;
        float* erow = pj.Ec + tok * pj.KP;
        const float sq = sq_sm[r_in_tile];
        float r2 = sq;
#pragma unroll 1
        for (int b0 = 0; b0 < nb0; b0 += 32) {
          float accv[32];
          {
            uint32_t g[32];
            tmem_ld32(tbase + b0, g);
#pragma unroll
            for (int i = 0; i < 32; ++i) accv[i] = __uint_as_float(g[i]);
          }
          const int b1 = min(nb0, b0 + 32);
          const bool full32 = b1 - b0 > 16;             // uniform: rows 16..31 of this chunk exist
#pragma unroll 1
          for (int qc = 0; qc < b0; qc += 8) {
            uint32_t ep[8];
            tmem_ld8(tbase + qc, ep);
            if (alive) {
#pragma unroll
              for (int qq = 0; qq < 8; qq += 4) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const float4 l = *reinterpret_cast<const float4*>(Lsm + (b0 + i) * BN + qc + qq);
                  accv[i] = fmaf(-l.x, __uint_as_float(ep[qq]), accv[i]);
                  accv[i] = fmaf(-l.y, __uint_as_float(ep[qq + 1]), accv[i]);
                  accv[i] = fmaf(-l.z, __uint_as_float(ep[qq + 2]), accv[i]);
                  accv[i] = fmaf(-l.w, __uint_as_float(ep[qq + 3]), accv[i]);
                }
                if (full32) {
#pragma unroll
                  for (int i = 16; i < 32; ++i) {
                    const float4 l = *reinterpret_cast<const float4*>(Lsm + (b0 + i) * BN + qc + qq);
                    accv[i] = fmaf(-l.x, __uint_as_float(ep[qq]), accv[i]);
                    accv[i] = fmaf(-l.y, __uint_as_float(ep[qq + 1]), accv[i]);
                    accv[i] = fmaf(-l.z, __uint_as_float(ep[qq + 2]), accv[i]);
                    accv[i] = fmaf(-l.w, __uint_as_float(ep[qq + 3]), accv[i]);
                  }
                }
              }
            }
          }
          // the triangle, in place: accv[i] becomes e_{b0+i}
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float v = 0.f;
            if (alive && b0 + i < b1) {
              v = accv[i];
#pragma unroll
              for (int q = 0; q < i; ++q) v = fmaf(-Lsm[(b0 + i) * BN + b0 + q], accv[q], v);
              v *= rinv_sm[b0 + i];
              r2 = fmaf(-v, v, r2);
            }
            accv[i] = v;
          }
          if (alive) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              if (b0 + i + 4 <= b1)
                *reinterpret_cast<float4*>(erow + b0 + i) = make_float4(accv[i], accv[i + 1], accv[i + 2], accv[i + 3]);
              else
                for (int u = i; u < b1 - b0 && u < i + 4; ++u) erow[b0 + u] = accv[u];
          }
          if (b0 + 32 < nb0) {
            uint32_t eb[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) eb[i] = __float_as_uint(accv[i]);
            tmem_st32(tbase + b0, eb);
          }
        }
        if (alive) {
          pj.r2[tok] = r2;
          pj.sqn[tok] = sq;
          pj.U[tok] = proj_value(__ldg(pj.scores + tok), r2, sq, pj.lambda, pj.tau);
          pj.cstep[tok] = nb0;
        }
      } else if constexpr (EPI == EPI_F32) {
        // products with per-image A rows write C at the same rows
        const long long orow = a.pr.n > 0 && a.pr.a_off && !a.pr.a_mn
                                   ? (__ldg(a.pr.a_off + c.b) + static_cast<long long>(row)) * a.ldc : crow;
        float* out = reinterpret_cast<float*>(q.C) + orow + col0 + c.ks * a.c_split_stride;
        const int ew = warp - 2;
#pragma unroll 1
        for (int ch = 0; ch < BN / 32; ++ch) {
          const int cbase = col0 + ch * 32;
          if (cbase >= lim) break;                       // uniform
          uint32_t r[32];
          tmem_ld32(tbase + ch * 32, r);
          if (a.box_store) {
            // 128-byte rows through shared memory (128-byte swizzle) to one box store, clipped at M and
            // N: written row by row from the lanes, a store instruction touches 32 rows, and a tile
            // took 6.8 us where this takes 2.5 us (the step of
            // 4 samples of 2880 tokens: 736 -> 699 us, 2 of 576: 245 -> 224 us)
            // (a tile stores an even number of chunks, so the two buffers alternate across tiles too)
            uint8_t* sb = stg + (ew * 2 + (ch & 1)) * 4096;
            if (lane == 0) bulk_wait_group_read<1>();    // this buffer's previous store has read it
            __syncwarp();
#pragma unroll
            for (int v = 0; v < 8; ++v)
              *reinterpret_cast<uint4*>(sb + lane * 128 + ((v ^ (lane & 7)) << 4)) =
                  make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_3d(&maps.C[0], sb, cbase, c.m_blk * kBM + lane_grp * 32, a.batch > 1 ? c.b : c.ks);
              bulk_commit_group();
            }
            continue;
          }
          if (row_ok && cbase < lim) {
            if (cbase + 32 <= lim) {
#pragma unroll
              for (int j = 0; j < 32; j += 4)
                *reinterpret_cast<float4*>(out + ch * 32 + j) =
                    make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]), __uint_as_float(r[j + 2]),
                                __uint_as_float(r[j + 3]));
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (cbase + j < lim) out[ch * 32 + j] = __uint_as_float(r[j]);
            }
          }
        }
      } else if constexpr (S::TSTORE) {
        // (hi, lo) of each 32x32 chunk go through shared memory to two TMA box stores
        // (coalesced, asynchronous); buffers alternate, reused once their store has read them
        const int ew = warp - 2;
        const int y = c.b * a.a_row_stride + c.m_blk * kBM + lane_grp * 32;   // first row of this warp
#pragma unroll 1
        for (int ch = 0; ch < BN / 32; ++ch) {
          const int cbase = col0 + ch * 32;
          if (cbase >= lim) break;                       // uniform: a last tile wider than what is left
          uint32_t r[32];
          tmem_ld32(tbase + ch * 32, r);
          uint8_t* hb = stg + (ew * 2 + (ch & 1)) * 4096;     // [hi 32x32 | lo 32x32] bf16
          if (lane == 0) bulk_wait_group_read<1>();      // this buffer's previous store has read it
          __syncwarp();
          uint32_t pk[16], pl[16];
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            float x0 = __uint_as_float(r[j]), x1 = __uint_as_float(r[j + 1]);
            if (q.bias) {
              const __nv_bfloat162 bb = __ldg(reinterpret_cast<const __nv_bfloat162*>(q.bias + cbase + j));
              x0 += __bfloat162float(bb.x);
              x1 += __bfloat162float(bb.y);
            }
            if constexpr (EPI == EPI_GELU_SPLIT) { x0 = gelu_erf(x0); x1 = gelu_erf(x1); }
            const __nv_bfloat162 hi = __floats2bfloat162_rn(x0, x1);
            pk[j / 2] = *reinterpret_cast<const uint32_t*>(&hi);
            pl[j / 2] = pack_bf16(x0 - __bfloat162float(hi.x), x1 - __bfloat162float(hi.y));
          }
          // 64-byte swizzle: 16-byte unit v of row r sits at unit v ^ ((r >> 1) & 3), so the
          // eight rows of a quarter warp hit distinct banks
          uint4* oh = reinterpret_cast<uint4*>(hb + lane * 64);
          uint4* ol = reinterpret_cast<uint4*>(hb + 2048 + lane * 64);
          const int sw = (lane >> 1) & 3;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            oh[v ^ sw] = make_uint4(pk[4 * v], pk[4 * v + 1], pk[4 * v + 2], pk[4 * v + 3]);
            ol[v ^ sw] = make_uint4(pl[4 * v], pl[4 * v + 1], pl[4 * v + 2], pl[4 * v + 3]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {                                 // rows past M are clipped by the store
            tma_store_2d(&maps.C[GROUPED ? c.grp : 0], hb, cbase, y);
            tma_store_2d(&maps.C[GROUPED ? c.grp : 0], hb + 2048, a.N + cbase, y);
            bulk_commit_group();
          }
        }
      } else {
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(q.C) + crow + col0;
#pragma unroll 1
        for (int ch = 0; ch < BN / 32; ++ch) {
          uint32_t r[32];
          tmem_ld32(tbase + ch * 32, r);
          const int cbase = col0 + ch * 32;
          if (row_ok && cbase < lim) {
            constexpr bool SPLIT = EPI == EPI_GELU_SPLIT || EPI == EPI_BIAS_SPLIT;
            uint32_t pk[16], pl[16];
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              float x0 = __uint_as_float(r[j]), x1 = __uint_as_float(r[j + 1]);
              if (q.bias) {
                const __nv_bfloat162 bb = __ldg(reinterpret_cast<const __nv_bfloat162*>(q.bias + cbase + j));
                x0 += __bfloat162float(bb.x);
                x1 += __bfloat162float(bb.y);
              }
              if constexpr (EPI == EPI_GELU_BF16 || EPI == EPI_GELU_SPLIT) { x0 = gelu_erf(x0); x1 = gelu_erf(x1); }
              const __nv_bfloat162 hi = __floats2bfloat162_rn(x0, x1);
              pk[j / 2] = *reinterpret_cast<const uint32_t*>(&hi);
              if constexpr (SPLIT) pl[j / 2] = pack_bf16(x0 - __bfloat162float(hi.x), x1 - __bfloat162float(hi.y));
            }
            uint4* o = reinterpret_cast<uint4*>(out + ch * 32);
#pragma unroll
            for (int v = 0; v < 4; ++v) o[v] = make_uint4(pk[4 * v], pk[4 * v + 1], pk[4 * v + 2], pk[4 * v + 3]);
            if constexpr (SPLIT) {
              uint4* ol = reinterpret_cast<uint4*>(out + a.N + ch * 32);
#pragma unroll
              for (int v = 0; v < 4; ++v) ol[v] = make_uint4(pl[4 * v], pl[4 * v + 1], pl[4 * v + 2], pl[4 * v + 3]);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (CG2) mbar_arrive_cluster(mapa_u32(&tempty[acc], 0));
        else mbar_arrive(S::PROJ ? sempty : &tempty[acc]);
      }
      if constexpr (S::PROJ) {
        acc_phase ^= 1;
      } else {
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1;
      }
    }
    if constexpr (S::TSTORE || S::TSTORE_F32) {
      if (lane == 0) bulk_wait_group_all();              // every box store has completed
      __syncwarp();
    }
  } else if constexpr (S::PROJ) {
    // ------------------------------------------------------------------ K slices' sums
    const int lane_grp = warp & 3;
    const uint32_t lanes = tmem_base + (static_cast<uint32_t>(lane_grp * 32) << 16);
    const int slices = min(SLICES, a.K / kBK);     // those with K blocks
    uint32_t acc = 0, acc_phase = 0, s_phase = 0;
    bool ok = true;
    for (int t = unit0; t < total && ok; t += units_step) {
      TileCoord c = coord(t);
      if (c.skip) continue;
      const int nb0 = min(BN, __ldg(a.proj.nbasis + c.b));
      float sum[BN], sq = 0.f;
#pragma unroll
      for (int j = 0; j < BN; ++j) sum[j] = 0.f;
#pragma unroll 1
      for (int sl = 0; sl < slices; ++sl) {
        if (!mbar_wait(&tfull[acc], acc_phase, a.status, abort_flag, a.wait_ns)) { ok = false; break; }
        tc_fence_after();
        float d = 0.f;                             // this row's diagonal element of A A^T
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
          uint32_t r[16];
          tmem_ld16(lanes + 3 * BN + lane_grp * 32 + h, r);
#pragma unroll
          for (int j = 0; j < 16; ++j) d = h + j == lane ? __uint_as_float(r[j]) : d;
        }
        sq += d;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(dempty);
#pragma unroll
        for (int ch = 0; ch < BN / 32; ++ch) {
          if (ch * 32 >= nb0) break;               // uniform
#pragma unroll
          for (int h = 0; h < 32; h += 16) {       // 16 at a time: 128 sums leave room for no more
            uint32_t r[16];
            tmem_ld16(lanes + acc * BN + ch * 32 + h, r);
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[ch * 32 + h + j] += __uint_as_float(r[j]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[acc]);
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1;
      }
      if (!ok || !mbar_wait(sempty, s_phase ^ 1, a.status, abort_flag, a.wait_ns)) break;
      tc_fence_after();
#pragma unroll
      for (int ch = 0; ch < BN / 32; ++ch) {
        if (ch * 32 >= nb0) break;                 // uniform
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(sum[ch * 32 + j]);
        tmem_st32(lanes + 2 * BN + ch * 32, r);
      }
      sq_sm[lane_grp * 32 + lane] = sq;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sfull);
      s_phase ^= 1;
    }
  }
  // Every role of this CTA has left its loop.  If one gave up (a bounded wait ran out), loads
  // may still be in flight that no MMA waited for: let them land before the CTA exits.  With
  // 2-SM pairs both CTAs' loads complete on the leader's barriers, which the leader drains.
  __syncthreads();
  if (*abort_flag && drains && crank == 0) {
    for (int s = 0; s < STAGES; ++s)
      if (last_par[s] >= 0) mbar_wait(&full[s], static_cast<uint32_t>(last_par[s]), a.status, nullptr);
  }
  if constexpr (PAIR) cluster_sync();             // no commit or remote arrive still in flight
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (CG2) tmem_dealloc_cg2(tmem_base, S::TMEM_COLS);
    else tmem_dealloc(tmem_base, S::TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2D bf16 tensor map over [rows, K] (K contiguous), box 64 x box_rows, 128-byte swizzle.
bool make_map(CUtensorMap* m, const void* base, long long rows, int K, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Tensor maps of one row group.
template <int BN, int EPI, bool PAIR, bool TSTORE>
bool make_maps(const GemmDesc& d, CUtensorMap& ta, CUtensorMap& tb, CUtensorMap& tc) {
  const bool prod = d.pr.n > 0;
  const int acols = prod ? d.pr.a_cols : (d.a_kwrap > 0 ? d.a_kwrap : d.K);
  const int bcols = prod ? d.pr.b_cols : d.K;
  if (!make_map(&ta, d.A, d.a_rows_total, acols, prod && d.pr.a_mn ? 64 : kBM)) return false;
  if (!make_map(&tb, d.B, d.b_rows_total, bcols, prod && d.pr.b_mn ? 64 : (PAIR ? BN / 2 : BN))) return false;
  tc = ta;
  if constexpr (TSTORE) {       // output [rows, ldc] bf16, 32x32 boxes, 64-byte swizzle
    // box stores clip at a_rows_total, which is the row bound M only for one flat batch
    if (d.batch != 1 || d.a_rows_total != d.M) return false;
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(d.ldc), static_cast<cuuint64_t>(d.a_rows_total)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(d.ldc) * 2};
    cuuint32_t box[2] = {32, 32};
    cuuint32_t estr[2] = {1, 1};
    if (fn(&tc, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, d.C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
        CUDA_SUCCESS)
      return false;
  }
  if constexpr (EPI == EPI_F32) {  // output [batch or ksplit][M][ldc] fp32, N columns, 32x32 boxes, 128-byte swizzle
    if (f32_box_store(d)) {
      auto fn = encode_fn();
      if (!fn) return false;
      const long long slice = d.batch > 1 ? d.c_batch_stride
                              : d.ksplit > 1 ? d.c_split_stride : static_cast<long long>(d.M) * d.ldc;
      cuuint64_t dims[3] = {static_cast<cuuint64_t>(d.N), static_cast<cuuint64_t>(d.M),
                            static_cast<cuuint64_t>(d.batch > 1 ? d.batch : d.ksplit)};
      cuuint64_t strides[2] = {static_cast<cuuint64_t>(d.ldc) * 4, static_cast<cuuint64_t>(slice) * 4};
      cuuint32_t box[3] = {32, 32, 1};
      cuuint32_t estr[3] = {1, 1, 1};
      if (fn(&tc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, d.C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
          CUDA_SUCCESS)
        return false;
    }
  }
  return true;
}

// d2: the second row group (predictor epilogues), or nullptr.
template <int BN, int STAGES, int EPI, bool PAIR = false>
cudaError_t run(const GemmDesc& d, const GemmDesc* d2, const KArgs& ka, int num_sms, cudaStream_t st) {
  using S = Smem<BN, STAGES, EPI, PAIR>;
  constexpr bool GROUPED = EPI == EPI_GELU_SPLIT || EPI == EPI_ROPE_SPLIT3;
  Maps maps;
  if (!make_maps<BN, EPI, PAIR, S::TSTORE>(d, maps.A[0], maps.B[0], maps.C[0])) return cudaErrorInvalidValue;
  if (!make_maps<BN, EPI, PAIR, S::TSTORE>(d2 ? *d2 : d, maps.A[1], maps.B[1], maps.C[1])) return cudaErrorInvalidValue;
  auto kern = gemm_tc_kernel<BN, STAGES, EPI, PAIR>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::TOTAL);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int n_tiles = (d.N + BN - 1) / BN, rows = PAIR ? 2 * kBM : kBM;
  int units = d.batch * ((d.M + rows - 1) / rows) * n_tiles * ka.ksplit;
  if (GROUPED) {
    units = 0;
    for (int g = 0; g < ka.groups; ++g) units += (ka.grp[g].M + rows - 1) / rows;   // the most there can be
    units *= n_tiles;
  }
  if (units == 0) return cudaSuccess;
  if (PAIR) {
    const int grid = 2 * std::max(1, std::min(units, num_sms / 2));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = S::TOTAL;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = pdl_disabled() ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, maps, ka);
  }
  const int grid = std::max(1, std::min(units, num_sms));
  return launch_k(kern, dim3(grid), dim3(S::THREADS), S::TOTAL, st, maps, ka);
}

// The fields of a row group.
RowGroup row_group(const GemmDesc& d) {
  RowGroup g{};
  g.M = d.M; g.C = d.C;
  g.bias = static_cast<const __nv_bfloat16*>(d.bias); g.biasf = d.biasf;
  g.pos = d.pos; g.pos_mod = d.pos_mod > 0 ? d.pos_mod : 1;
  g.split_kind = d.split_kind; g.scale = d.scale; g.aux = d.aux;
  g.seg_valid = d.seg_valid; g.seg_len = d.seg_len;
  return g;
}

}  // namespace

// Columns of the first predictor layer's 2-SM tiles (256 rows of either branch, one launch): the
// width with the least time by the model
//   waves of the tiles over the SM pairs x K blocks x the longer of the MMA (2 BN cycles) and the
//   copies into an SM (256 + BN), and the last tile's epilogue (40 BN).
// Large batches take 256.  With few rows the chip would idle behind a few wide tiles, each a chain of
// K / 64 blocks: 576 visual and 32 question rows take 64 (64 pairs instead of 16).  The width changes
// no sum.
int predictor_tile_width(long long m_vis, long long m_text, int N, int K, int num_sms) {
  const long long pairs = std::max(1, num_sms / 2);
  const long long rows = (m_vis + 2 * kBM - 1) / (2 * kBM) + (m_text + 2 * kBM - 1) / (2 * kBM);
  long long best = -1;
  int width = 256;
  for (int bn : {256, 192, 128, 64}) {
    const long long units = rows * ((N + bn - 1) / bn);
    const long long t = (units + pairs - 1) / pairs * (K / kBK) * std::max(2 * bn, 256 + bn) + 40 * bn;
    if (best < 0 || t < best) {
      best = t;
      width = bn;
    }
  }
  return width;
}

namespace {
cudaError_t check_desc(const GemmDesc& d);
cudaError_t launch_checked(const GemmDesc& d, const GemmDesc* d2, int num_sms, cudaStream_t st);
}  // namespace

cudaError_t launch_gemm(const GemmDesc& d, int num_sms, cudaStream_t st) {
  const cudaError_t e = check_desc(d);
  if (e != cudaSuccess) return e;
  return d.M == 0 ? cudaSuccess : launch_checked(d, nullptr, num_sms, st);
}

cudaError_t launch_gemm_groups(const GemmDesc& d, const GemmDesc& d2, int num_sms, cudaStream_t st) {
  cudaError_t e = check_desc(d);
  if (e == cudaSuccess) e = check_desc(d2);
  if (e != cudaSuccess) return e;
  // what the groups share, and what only one group has
  if ((d.epi != EPI_GELU_SPLIT && d.epi != EPI_ROPE_SPLIT3) || d2.epi != d.epi || d2.N != d.N || d2.K != d.K ||
      d2.ldc != d.ldc || d2.a_kwrap != d.a_kwrap || d2.split3 != d.split3 || d2.rope != d.rope ||
      d2.rope_ld != d.rope_ld || d2.tile_n != d.tile_n || d2.wait_ns != d.wait_ns || d2.status != d.status ||
      d.batch != 1 || d2.batch != 1 || d.M == 0 || d2.M == 0)
    return cudaErrorInvalidValue;
  return launch_checked(d, &d2, num_sms, st);
}

namespace {
cudaError_t check_desc(const GemmDesc& d) {
  if (d.K <= 0 || d.K % kBK != 0 || d.M < 0 || d.N <= 0 || d.batch <= 0) return cudaErrorInvalidValue;
  if (d.a_kwrap < 0 || d.a_kwrap % kBK != 0 || d.a_kwrap > d.K) return cudaErrorInvalidValue;
  if (d.split3 && (d.K % (3 * kBK) != 0 || d.a_kwrap != 2 * (d.K / 3))) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(d.A) | reinterpret_cast<uintptr_t>(d.B)) & 15) return cudaErrorInvalidValue;
  // every output row and column block is written with 16-byte vector stores
  const bool scalar_out = d.epi == EPI_SM_STATS || d.epi == EPI_SM_MEAN;   // float / float2 stores
  const bool f32 = d.epi == EPI_F32 || d.epi == EPI_ROPE_F32;
  const long long vec = f32 ? 4 : 8;
  if (d.epi == EPI_PROJECT) {      // writes through ProjArgs only (float4 reads of Ec rows)
    if (d.proj.KP % 4 != 0 || !d.proj.Ec || (reinterpret_cast<uintptr_t>(d.proj.Ec) & 15)) return cudaErrorInvalidValue;
  } else if (!scalar_out &&
             (d.ldc % vec != 0 || d.c_batch_stride % vec != 0 || (reinterpret_cast<uintptr_t>(d.C) & 15))) {
    return cudaErrorInvalidValue;
  }
  if (scalar_out && (!d.stats || (reinterpret_cast<uintptr_t>(d.stats) & 7) || (reinterpret_cast<uintptr_t>(d.C) & 3)))
    return cudaErrorInvalidValue;
  if ((d.epi == EPI_GELU_SPLIT || d.epi == EPI_BIAS_SPLIT) && d.ldc < 2LL * d.N) return cudaErrorInvalidValue;
  // split-K: fp32 partial tiles only, every slice at least one K block
  if (d.ksplit < 1 || (d.ksplit > 1 && (d.epi != EPI_F32 || d.ksplit > d.K / kBK || d.c_split_stride % 4 != 0)))
    return cudaErrorInvalidValue;
  if (d.blist && !d.bcount) return cudaErrorInvalidValue;
  if (d.pr.n) {      // segments start at whole boxes; K is the products' K blocks side by side
    const GemmProducts& q = d.pr;
    if (d.epi != EPI_F32 || q.n < 0 || q.n > kMaxProducts || d.a_kwrap || d.split3 || d.b_off || d.b_base ||
        q.kblocks <= 0 || d.K != q.n * q.kblocks * kBK || q.a_cols % 8 != 0 || q.b_cols % 8 != 0)
      return cudaErrorInvalidValue;
    for (int i = 0; i < q.n; ++i)
      if (q.a_seg[i] < 0 || q.a_seg[i] % kBK != 0 || q.b_seg[i] < 0 || q.b_seg[i] % kBK != 0)
        return cudaErrorInvalidValue;
  }
  if (d.seg_valid && (d.seg_len < 1 || d.batch != 1 || (d.epi != EPI_GELU_SPLIT && d.epi != EPI_ROPE_SPLIT3)))
    return cudaErrorInvalidValue;
  return cudaSuccess;
}

cudaError_t launch_checked(const GemmDesc& d, const GemmDesc* d2, int num_sms, cudaStream_t st) {
  KArgs ka;
  ka.grp[0] = row_group(d);
  ka.grp[1] = row_group(d2 ? *d2 : d);
  ka.groups = d2 ? 2 : 1;
  ka.M = d.M; ka.N = d.N; ka.K = d.K; ka.batch = d.batch;
  ka.a_row_stride = d.a_row_stride; ka.b_row_stride = d.b_row_stride;
  ka.n_limit = d.n_limit; ka.ldc = d.ldc; ka.c_batch_stride = d.c_batch_stride;
  ka.rope = d.rope; ka.rope_half = d.rope_half; ka.rope_ld = d.rope_ld;
  ka.status = d.status;
  ka.b_off = d.b_off;
  ka.stats = d.stats; ka.stat_ld = d.stat_ld; ka.stat_parts = d.stat_parts; ka.col_count = d.col_count;
  ka.b_base = d.b_base; ka.proj = d.proj;
  ka.a_kwrap = d.a_kwrap; ka.split3 = d.split3;
  ka.blist = d.blist; ka.bcount = d.blist ? d.bcount : nullptr;
  ka.m_limit = d.m_limit;
  ka.wait_ns = d.wait_ns > 0 ? static_cast<unsigned long long>(d.wait_ns) : kWaitLimitNs;
  ka.ksplit = d.ksplit; ka.c_split_stride = d.c_split_stride;
  ka.box_store = f32_box_store(d);
  ka.pr = d.pr;
  switch (d.epi) {
    case EPI_GELU_BF16:
      if (d.N % 256 == 0) return run<256, 4, EPI_GELU_BF16>(d, d2, ka, num_sms, st);
      if (d.N % 64 == 0) return run<64, 8, EPI_GELU_BF16>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_BIAS_BF16:
      if (d.N % 256 == 0) return run<256, 4, EPI_BIAS_BF16>(d, d2, ka, num_sms, st);
      if (d.N % 64 == 0) return run<64, 8, EPI_BIAS_BF16>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_ROPE_F32:
      if (d.N == 64) return run<64, 8, EPI_ROPE_F32>(d, d2, ka, num_sms, st);
      if (d.N == 128) return run<128, 6, EPI_ROPE_F32>(d, d2, ka, num_sms, st);
      if (d.N == 256) return run<256, 4, EPI_ROPE_F32>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_GELU_SPLIT:
      if (d.N % 256 == 0) {
        switch (d.tile_n) {
          case 64: return run<64, 8, EPI_GELU_SPLIT, true>(d, d2, ka, num_sms, st);
          case 128: return run<128, 8, EPI_GELU_SPLIT, true>(d, d2, ka, num_sms, st);
          case 192: return run<192, 6, EPI_GELU_SPLIT, true>(d, d2, ka, num_sms, st);
          default: return run<256, 6, EPI_GELU_SPLIT, true>(d, d2, ka, num_sms, st);
        }
      }
      if (d.N % 64 == 0) return run<64, 8, EPI_GELU_SPLIT>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_BIAS_SPLIT:
      if (d.N % 256 == 0) return run<256, 6, EPI_BIAS_SPLIT, true>(d, d2, ka, num_sms, st);
      if (d.N % 64 == 0) return run<64, 8, EPI_BIAS_SPLIT>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_ROPE_SPLIT3:   // dp = 128: 2-SM pairs share the B tile (each CTA loads 64 of its rows)
      if (d.N == 64) return run<64, 8, EPI_ROPE_SPLIT3>(d, d2, ka, num_sms, st);
      if (d.N == 128) return run<128, 8, EPI_ROPE_SPLIT3, true>(d, d2, ka, num_sms, st);
      return cudaErrorInvalidValue;
    case EPI_SM_STATS:
      return run<256, 4, EPI_SM_STATS>(d, d2, ka, num_sms, st);
    case EPI_SM_MEAN:
      return run<256, 4, EPI_SM_MEAN>(d, d2, ka, num_sms, st);
    case EPI_PROJECT:
      if (d.N > kProjMaxBasis || d.batch < 1) return cudaErrorInvalidValue;
      if (d.N <= 32) return run<32, 8, EPI_PROJECT>(d, d2, ka, num_sms, st);
      if (d.N <= 96) return run<96, 6, EPI_PROJECT>(d, d2, ka, num_sms, st);
      return run<128, 5, EPI_PROJECT>(d, d2, ka, num_sms, st);
    case EPI_F32:   // the distillation's contractions
      if (d.M <= kBM && d.N <= 128) return run<128, 6, EPI_F32>(d, d2, ka, num_sms, st);
      return run<256, 6, EPI_F32, true>(d, d2, ka, num_sms, st);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace

}  // namespace mapk
