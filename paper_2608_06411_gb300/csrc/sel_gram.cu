// Gram blocks of the selection, G = Va Vb^T in fp32, for the rows of an image's active slots
// against themselves and against its basis tokens: <v_i, v_j> of Eq. 4's residuals.
//
// A block is 256 rows by at most 256, from up to 3 MB of scattered feature rows, so one SM (or a
// 2-SM pair) would spend 15 to 25 us on the copies alone at the 40-odd bytes a cycle an SM takes
// in.  A cluster of 8 CTAs splits K instead: each copies its eighth of every row straight from the
// features by slot (no gathered copy in between), multiplies on its own tensor core, and the eight
// partial blocks are added through distributed shared memory, in rank order (the same sums
// whatever the batch).  Per CTA:
//   all threads   cp.async rows (16 bytes a thread, 128 bytes of a row per 8 threads) into a ring
//                 of 128-byte-swizzled K-major stages of 64 columns;
//   one thread    tcgen05.mma (M = 128, K = 16) per stage into TMEM: columns 0-127 the rows 0-127,
//                 the next ones the rows 128-255;
//   all threads   TMEM -> shared memory (the ring's space), cluster barrier, an eighth of the rows
//                 summed over the ranks and written.
// Active by active is symmetric: only the tiles at and below the diagonal are computed.
// The gathered copy and a one-CTA or one-pair GEMM took 25 us for G[R0, R0] and 33 us for a round's
// block of one image of 2880 x 4096; with this kernel the call went from 313 to 274 us (576 tokens:
// 228 to 190, 64 images 2173 to 2141, k = 640 of 2 images 1535 to 1291).
#include "kernels.h"
#include "ptx.cuh"
#include "select.h"

namespace mapk {
namespace {

constexpr int kRanks = kGramSlices;                  // CTAs of a cluster, a K slice each
constexpr int kThreads = 256;
constexpr int kTileRows = 128;
constexpr int kKb = 64;                              // columns of a stage
constexpr int kBasisCols = kGramBasisCols;           // basis tokens per unit
static_assert(kActiveSlots == 2 * kTileRows && kBasisCols == kTileRows, "tiles of 128 x 128");

constexpr uint32_t kRowBytes = kKb * 2;
constexpr uint32_t kActBytes = kActiveSlots * kRowBytes, kBasBytes = kBasisCols * kRowBytes;
constexpr uint32_t kRingBytes = 6 * kActBytes;       // 6 stages of active rows, or 4 with basis rows
constexpr uint32_t kTileFloats = kTileRows * kTileRows;
static_assert(4 * (kActBytes + kBasBytes) <= kRingBytes && 3 * kTileFloats * 4 <= kRingBytes, "ring, then partial tiles");
constexpr uint32_t kSmem = kRingBytes + 1024;

// 16-byte asynchronous copy, or 16 zero bytes.
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

struct Shared {
  uint64_t empty[6], done;
  uint32_t tmem;
  int abort;
};

// This CTA's K slice of one unit, accumulated in TMEM.  BASIS: active rows x basis rows, else the
// active rows' tiles at and below the diagonal (two: false when rows 128.. are empty).
template <bool BASIS>
__device__ __forceinline__ void multiply(const SelState& s, int b, const int (&ta)[8], const int (&tb)[4], bool two,
                                         uint32_t ring, Shared& sh, uint32_t tmem, int kb0, int kb1,
                                         unsigned long long wait_ns) {
  constexpr int STAGES = BASIS ? 4 : 6, LAG = STAGES - 2;
  constexpr uint32_t STAGE = kActBytes + (BASIS ? kBasBytes : 0);
  const int tid = threadIdx.x, r0 = tid >> 3, c = tid & 7;
  const bool warp0 = __shfl_sync(0xffffffffu, tid >> 5, 0) == 0;
  const uint16_t* V = static_cast<const uint16_t*>(s.uptr ? s.uptr[1] : s.V) + static_cast<long long>(b) * s.N * s.D + 8 * c;
  const int n = kb1 - kb0;
  volatile int* abort_flag = &sh.abort;
  for (int it = 0; it < n + LAG; ++it) {
    if (it < n) {
      const int st = it % STAGES;
      if (it >= STAGES) mbar_wait(&sh.empty[st], ((it / STAGES) - 1) & 1, s.status, abort_flag, wait_ns);
      const uint32_t base = ring + st * STAGE;
      const long long col = static_cast<long long>(kb0 + it) * kKb;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = r0 + 32 * i;
        if (i < 4 || two)
          cp_async16_or_zero(base + r * kRowBytes + ((c ^ (r & 7)) << 4),
                             V + static_cast<long long>(ta[i] < 0 ? 0 : ta[i]) * s.D + col, ta[i] >= 0);
      }
      if (BASIS) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = r0 + 32 * i;
          cp_async16_or_zero(base + kActBytes + r * kRowBytes + ((c ^ (r & 7)) << 4),
                             V + static_cast<long long>(tb[i] < 0 ? 0 : tb[i]) * s.D + col, tb[i] >= 0);
        }
      }
    }
    cp_async_commit();
    if (it >= LAG) {
      cp_async_wait_group<LAG>();                    // this thread's copies of K block it - LAG
      fence_proxy_async_smem();                      // visible to the tensor core's reads
      __syncthreads();
      if (warp0 && elect_one() && !*abort_flag) {
        tc_fence_after();
        const int j = it - LAG, st = j % STAGES;
        const uint32_t a0 = ring + st * STAGE, a1 = a0 + kTileRows * kRowBytes, bb = a0 + kActBytes;
        const uint64_t d0 = desc_sw128(0) + (a0 >> 4), d1 = desc_sw128(0) + (a1 >> 4), db = desc_sw128(0) + (bb >> 4);
#pragma unroll
        for (int k = 0; k < kKb / 16; ++k) {
          const uint32_t on = j != 0 || k != 0;
          if (BASIS) {
            umma_bf16(tmem, d0 + 2 * k, db + 2 * k, idesc_bf16(128, 128), on);
            if (two) umma_bf16(tmem + 128, d1 + 2 * k, db + 2 * k, idesc_bf16(128, 128), on);
          } else {
            umma_bf16(tmem, d0 + 2 * k, d0 + 2 * k, idesc_bf16(128, 128), on);
            if (two) umma_bf16(tmem + 128, d1 + 2 * k, d0 + 2 * k, idesc_bf16(128, 256), on);
          }
        }
        umma_commit(&sh.empty[st]);
      }
    }
  }
}

// Grid (kRanks, units, B), clusters of kRanks: unit 0 the active rows (the first `rows` slots)
// against themselves, unit u > 0 against basis tokens gbase + 128 (u - 1) ... of the image.
__global__ void __launch_bounds__(kThreads, 1) sel_gram_kernel(SelState s, int rows, unsigned long long wait_ns) {
  pdl_enter();
  const int b = blockIdx.z, unit = blockIdx.y, rank = static_cast<int>(cluster_ctarank());
  if (s.done[b]) return;                             // uniform in the cluster
  const int S = s.S, gbase = s.gbase[b], nbas = s.nbasis[b] - gbase;
  const int c0 = (unit - 1) * kBasisCols;
  if (unit > 0 && c0 >= nbas) return;
  extern __shared__ uint8_t raw[];
  __shared__ Shared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t ring = (smem_u32(raw) + 1023u) & ~1023u;
  float* part = reinterpret_cast<float*>(raw + (ring - smem_u32(raw)));
  if (tid == 0) {
    for (int i = 0; i < 6; ++i) mbar_init(&sh.empty[i], 1);
    mbar_init(&sh.done, 1);
    sh.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem, 512);
    tmem_relinquish();
  }
  int ta[8], tb[4];                                  // tokens of this thread's rows (-1: none)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = (tid >> 3) + 32 * i;
    ta[i] = r < rows ? s.aslot[static_cast<long long>(b) * S + r] : -1;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int q = c0 + (tid >> 3) + 32 * i;
    tb[i] = unit > 0 && q < nbas ? s.basis_tok[static_cast<long long>(b) * s.K + gbase + q] : -1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem;
  const bool two = rows > kTileRows;
  const int KB = s.D / kKb, kb0 = rank * KB / kRanks, kb1 = (rank + 1) * KB / kRanks;
  if (unit > 0) multiply<true>(s, b, ta, tb, two, ring, sh, tmem, kb0, kb1, wait_ns);
  else multiply<false>(s, b, ta, tb, two, ring, sh, tmem, kb0, kb1, wait_ns);
  if (kb1 > kb0) {                                   // every MMA has read its stage and written TMEM
    if (warp == 0 && elect_one()) umma_commit(&sh.done);   // by the thread that issued them
    mbar_wait(&sh.done, 0, s.status, nullptr);
    tc_fence_after();
  }
  __syncthreads();
  // partial tiles: rows of 128 floats, 16-byte units exchanged by the row's low bits
  const int tiles = unit > 0 ? (two ? 2 : 1) : (two ? 3 : 1);
  {
    const int g = warp & 3, r = g * 32 + lane, chunks = tiles * 4;   // chunks of 32 columns
    for (int ch = warp >> 2; ch < chunks; ch += 2) {
      uint32_t x[32];
      tmem_ld32(tmem + (static_cast<uint32_t>(g * 32) << 16) + ch * 32, x);
      float4* row = reinterpret_cast<float4*>(part) + ((ch >> 2) * kTileRows + r) * 32;
      const bool any = kb1 > kb0;                    // an empty K slice adds nothing
#pragma unroll
      for (int v = 0; v < 8; ++v)
        row[((ch & 3) * 8 + v) ^ (r & 7)] =
            any ? make_float4(__uint_as_float(x[4 * v]), __uint_as_float(x[4 * v + 1]), __uint_as_float(x[4 * v + 2]),
                              __uint_as_float(x[4 * v + 3]))
                : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  tc_fence_before();
  cluster_sync();                                    // every rank's partial tiles are written
  {
    uint32_t peer[kRanks];
#pragma unroll
    for (int p = 0; p < kRanks; ++p) peer[p] = mapa_u32(part, p);
    float* G = s.G + static_cast<long long>(b) * S * s.R;
    const int nrows = tiles * kTileRows / kRanks;
    for (int i = warp; i < nrows; i += kThreads / 32) {
      const int pr = rank * nrows + i, tile = pr / kTileRows, r = pr - tile * kTileRows;
      const uint32_t off = (pr * 32 + (lane ^ (r & 7))) * 16;
      float4 v[kRanks];
#pragma unroll
      for (int p = 0; p < kRanks; ++p) v[p] = ld_cluster_f4(peer[p] + off);
      float4 a = v[0];
#pragma unroll
      for (int p = 1; p < kRanks; ++p) { a.x += v[p].x; a.y += v[p].y; a.z += v[p].z; a.w += v[p].w; }
      // tile -> block: active x active (0, 0), (1, 0), (1, 1); active x basis (0, .), (1, .)
      const int gr = (unit > 0 ? tile : (tile > 0 ? 1 : 0)) * kTileRows + r;
      const int gc = (unit > 0 ? S + c0 : (tile == 2 ? kTileRows : 0)) + 4 * lane;
      if (gc + 4 <= s.R) *reinterpret_cast<float4*>(G + static_cast<long long>(gr) * s.R + gc) = a;
    }
  }
  cluster_sync();                                    // no rank leaves while a peer may read its tiles
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

cudaError_t launch_sel_gram(const SelState& s, int rows, int basis, long long wait_ns, cudaStream_t st) {
  if (s.S != kActiveSlots || rows < 1 || rows > s.S || basis < 0 || s.D % kKb != 0 || s.R % 4 != 0)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(sel_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmem));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kRanks, 1 + (basis + kBasisCols - 1) / kBasisCols, s.B);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kRanks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = pdl_disabled() ? 0 : 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, sel_gram_kernel, s, rows,
                            wait_ns > 0 ? static_cast<unsigned long long>(wait_ns) : kWaitLimitNs);
}

}  // namespace mapk
