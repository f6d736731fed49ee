// tbn_conv_igemm.cuh -- the tcgen05 implicit-GEMM kernel of the two-bit
// convolution (Eq. 1, Section 2) and its launch, shared by the translation
// units that instantiate it (tbn_conv_igemm.cu: host dispatch, the gathering
// and space-to-depth modes; tbn_conv_igemm_tma64.cu / _tma32.cu: the TMA modes
// with and without fused quantization; tbn_conv_igemm_pair.cu: tap pairs;
// tbn_conv_igemm_pad.cu: padded channels and row pairs), so that its variants compile in parallel.
//
//
// GEMM view of one tile:  D[128 filters x T pixels] = A[128 x n] * B[n x T]
// with T <= 256 output pixels and n = R*S*C in the codes' (r, s, c) order,
// 64 codes per K block (= pipeline stage: four MMAs of K = 16).
//
//   A (filters)     the 2-bit codes, decoded in registers to bf16 W~/2 in
//                   {+-0.5, +-1} (exact) and written straight into tensor
//                   memory (tcgen05.st) by eight "expander" warps: two per
//                   TMEM sub-partition, each decoding half of a K block's 64
//                   codes for the 32 filter rows (= TMEM lanes) it can reach,
//                   two K blocks per tcgen05.wait::st.  The decoded weights
//                   never touch shared memory, which is left to the
//                   activation operand.  Decoding costs integer-pipe issue
//                   slots per (filter, code), so a tile spans up to 256
//                   pixels to amortize it over as many MMA columns as the
//                   instruction allows.
//   B (activations) im2col rows per pixel, 128-byte rows (64 codes) with the
//                   128-byte swizzle.  When C % 64 == 0 a K block is one tap x
//                   64 channels and one TMA box load fetches it (the box is
//                   the tile's output pixels shifted by the tap; zero fill
//                   supplies the padding, element strides the conv stride).
//                   A tile is a run of consecutive output pixels of the
//                   whole batch, fetched in im2col mode, or whole output
//                   rows, fetched as a tiled box (see plan_conv).
//                   When C % 32 == 0 (e.g. 96 channels) a K block is two
//                   boxes of 32 channels, each from its own tap, into two
//                   64-byte-row halves of the stage with the 64-byte swizzle
//                   (a box past the filter's last code is loaded out of
//                   range and arrives zero-filled); on the widest tiles two
//                   taps share such a block for their last 32 channels and
//                   have 64-channel boxes before it (kModeTapPair).  When
//                   C % 8 == 0 (other
//                   counts) every tap has ceil(C / 64) K blocks of its own:
//                   the last box of a tap reaches past C and arrives
//                   zero-filled there, so whatever codes stand in those
//                   columns add zero, and whole steps of 16 past C are
//                   skipped (8 and 24 channels: see pad_boxes_pay).
//                   Otherwise gather warps assemble the rows from
//                   a per-K-block table of (tap, channel) offsets.
//   D               fp32 in tensor memory (256 columns).  Epilogue warps read
//                   lane = filter, column = pixel, multiply by 2 * alpha (Eq. 1
//                   applies alpha to the whole filter; the factor 2 undoes the
//                   W~/2 encoding -- exact scalings), add the optional
//                   residual (loaded by TMA to where its outputs are staged),
//                   apply ReLU and the optional 2x2 max pool, round to bf16
//                   into a shared-memory staging tile laid out as the NHWC
//                   output box, and TMA tensor stores write the box (clipped
//                   at the tensor's edges).  The accumulator is
//                   released as soon as it has been read, before the staging
//                   writes and the store complete.
//
// The kernel is persistent: each CTA walks tiles blockIdx.x, +gridDim.x, ...
// (filter tile fastest, so CTAs working at the same time share activation
// tiles in L2); producers and expanders run ahead into the next tile while
// the epilogue drains the accumulator.
//
// Warp roles (every role is a whole warp that waits on the barriers; where a
// single thread must issue -- TMA copies, MMAs, commits -- one elected lane
// does, with warp-uniform operands):
//   warps 0, 18.. TMA producers (TMA mode), taking K blocks in turn: one
//                 issuing thread delivers tiled boxes at a limited rate, so
//                 several keep the activation ring fuller
//   warp 1        TMEM allocator + MMA issuer
//   warps 2-9     expanders (in space-to-depth mode, done with the filter
//                 after the first tile, they join the epilogue)
//   warps 10-17   epilogue
//   warps 18-21   gather producers (gather mode only)
// Every wait is bounded (tbn_device.cuh); on a timeout the CTA records the
// error, drains its own in-flight copies and MMAs, frees TMEM and returns.
//
// The kernel is launched as a programmatic dependent of the previous kernel
// on the stream: its start-up (TMEM allocation, barrier set-up, tables) may
// overlap the previous kernel's last wave.  Every role passes
// grid_dependency_wait() before its first global read or write: only behind
// that wait are the previous kernel's writes visible, and the codes may be
// among them (a quantizer, or the transposition of the backward pass).  Each
// CTA lets its own dependents start once it has passed its wait, so
// everything older than the previous kernel is complete by then.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "tbn_device.cuh"
#include "tbn_internal.h"
#include "tbn_quant_core.cuh"

namespace tbn {

// The kernel's arguments and tile plan (plain data; built on the host by
// launch_conv_igemm).
struct IgArgs {
  int N, C, H, W, K, R, S, sh, sw, ph, pw, P, Q;
  int bw, bh, bn;          // output pixels per tile along q, p, image
  int tile_n;              // MMA N: bw*bh*bn rounded up to 16
  int tiles_q, tiles_p, tiles_k, tiles;
  int kblocks;             // ceil(R*S*C / 64): pipeline stages per tile
  int ncodes;              // R*S*C
  int wpf;                 // words per filter
  const __nv_bfloat16* x;  // gather mode
  const uint32_t* codes;
  const float* alpha;
  void* y;
  const void* residual;
  int relu, y_bf16;
  uint32_t* err;
  // im2col tiles: N, P and Q above are the extents that the tiles walk (the
  // batch as one row of N P Q pixels, or as one image of N P rows when
  // pooling); an image's output is iP x iQ
  int im2col, iP, iQ;
  // divisors of the tile and pixel coordinates
  FastDiv by_base /* by ksplit with clusters */, by_k, by_tq, by_tp, by_iq, by_ip;
  // patch mode: the patch is rows [p0 sh - ph, + PR) x columns [-pw, W + pw)
  int PR, PW;              // patch rows, patch columns (W + 2 pw)
  int patch_cap;           // bytes per patch buffer (multiple of 16)
  int patch_bulk;          // pw == 0: in-image rows are one contiguous range of x
  long long x_bytes;       // size of x (bulk copies never read past it)
  // split K: tile t is K-block range `split` (t / base_tiles) of the output
  // tile t % base_tiles; the fp32 partial sums go to `partial`
  // [ksplit][N][P][Q][K] and a second kernel adds them in split order
  int ksplit, kb_per, base_tiles;
  // or, in clusters of ksplit CTAs (CTA i: K-block range i % ksplit of output
  // tile i / ksplit), the cluster adds them itself (add_cluster_sums)
  int cluster;
  // two accumulators (tile_n <= 176): tile i accumulates into columns
  // [176 (i % 2), + 176), so its MMAs need not wait for the epilogue of
  // tile i - 1; the weight ring then starts at column 352
  int acc2;
  float* partial;
  // space-to-depth mode: the convolution in original coordinates (stride
  // s2d_s, C0 channels, R0 x S0 filter, codes in (r, s, c) order)
  int s2d_s, s2d_C, s2d_R, s2d_S;
  // fused quantization (Algorithm 1's quantization loop in the same launch):
  // the CTAs first write codes and alpha from the fp32 filters wq
  // [K][ncodes], then meet at a grid-wide barrier (a cooperative launch)
  // before convolving; null wq: codes and alpha are inputs
  const float* wq;
  uint32_t* codes_w;       // = codes
  float* alpha_w;          // = alpha
  unsigned* gbar;          // barrier word, zero at launch
  int wq_vec;              // 16-byte loads of wq allowed
};

struct TilePlan {
  int bw, bh, bn, T, tile_n, tiles_q, tiles_p, tiles_n;
  bool im2col;             // tiles of consecutive pixels over the whole batch
  bool rowpair;            // two output rows' filters in the MMA's 128 rows (kModeRowPair)
  int64_t oN, oP, oQ;      // output extents that the tiles walk
};

namespace {


constexpr int kBM = 128;            // filters per tile = TMEM lanes
constexpr int kBK = 64;             // codes per K block (128-byte rows)
constexpr int kMaxTileN = 256;      // pixels per tile (MMA N) upper bound
constexpr int kStages = 5;          // pipeline depth: activation ring (shared
                                    // memory) and weight ring (tensor memory)
constexpr int kAColsPerStage = kBK / 2;   // 64 bf16 = 32 columns of 32 bits
constexpr int kAccCols = kMaxTileN;       // the accumulator
constexpr int kAcc2Cols = 176;            // each of two accumulators (tiles of <= 176 pixels)
constexpr int kTmemCols = 512;      // accumulator [0,256) + weight ring [256,416)
constexpr int kExpWarps = 8;
constexpr int kEpiWarps = 8;
constexpr int kGatherWarps = 4;
constexpr int kPatchWarps = 8;      // patch mode: one operand row per thread
constexpr int kTmaProducers = 2;    // TMA mode: warp 0 and warps 18 .. 18 + kTmaProducers - 2
static_assert(kTmaProducers <= kStages, "a producer's parity wait needs kStages >= producers");
constexpr int kFirstExpWarp = 2;
constexpr int kFirstEpiWarp = kFirstExpWarp + kExpWarps;
constexpr int kFirstGatherWarp = kFirstEpiWarp + kEpiWarps;
constexpr int kStageBytes = kMaxTileN * kBK * 2;     // 32 KiB
constexpr int kOutStageBytes = kMaxTileN * kBM * 2;  // 64 KiB bf16 output box
constexpr uint64_t kWaitLimitNs = 1000000000ull;    // 1 s
constexpr int kMaxCluster = 8;      // K ranges of a cluster (the portable cluster size)

static_assert(kAccCols + kStages * kAColsPerStage <= kTmemCols, "TMEM budget");
static_assert(2 * kAcc2Cols + kStages * kAColsPerStage <= kTmemCols, "TMEM budget");

// How the activation operand reaches the stage ring.
constexpr int kModeTma64 = 0;   // one 64-channel TMA box per K block (C % 64 == 0)
constexpr int kModeTma32 = 1;   // two 32-channel TMA boxes per K block (C % 32 == 0)
constexpr int kModeGather = 2;  // threads gather each code's activation from global memory
constexpr int kModePatch = 3;   // the tile's input rows are staged in shared memory (bulk
                                // copy, double-buffered) and threads build the rows from there
constexpr int kModeS2d = 4;     // space-to-depth input: 64-channel TMA boxes, and the
                                // filter's K blocks decoded once per CTA into tensor memory
constexpr int kModeTmaPad = 5;  // 64-channel TMA boxes, each tap's last one padded (C % 8 == 0)
// Row pairs (K <= 64 filters, stride 1): MMA rows 0-63 are the filters for the
// even output rows, rows 64-127 the same filters, one tap row later, for the
// odd ones.  Both read the same box of input rows 2 i + r', r' = 0 .. R, so
// R + 1 tap rows serve two output rows where one at a time takes 2 R with
// half the MMA's rows empty.  The first tap row is the even rows' alone and
// the last the odd rows': their MMAs leave the other half's accumulators as
// they are (disabled output lanes), so an infinite or NaN input reaches the
// outputs whose taps read it and no others, at no cost.
constexpr int kModeRowPair = 6;
// Tap pairs (C = 64 m + 32, m >= 1): the K blocks of two taps are each tap's m
// whole 64-channel boxes, then one block of both taps' last 32 channels, so
// that 4 m + 2 boxes of 64-byte rows become 2 m boxes of 128-byte rows and two
// of 64: the boxes' rows are what paces wide tiles (see tap_pairs_pay).
constexpr int kModeTapPair = 7;
constexpr int kMaxResidentKB = 15;   // resident K blocks: up to 32 columns each beside the accumulator

__host__ __device__ constexpr bool mode_gathers(int mode) {
  return mode == kModeGather || mode == kModePatch;
}
// the patch buffers take the room of two ring stages
__host__ __device__ constexpr int stages_for(int mode) { return mode == kModePatch ? kStages - 2 : kStages; }

// Producer warps of a mode (warps kFirstGatherWarp.. in the gathering modes).
__host__ __device__ constexpr int producer_warps(int mode) {
  return mode == kModePatch ? kPatchWarps : (mode == kModeGather ? kGatherWarps : 0);
}

// Epilogue warps of a mode: in space-to-depth mode the expanders, done with
// the filter after the first tile, join them (the one accumulator is held for
// half as long: AlexNet conv1 at batch 256, 9 K blocks per tile, spent 30% of
// its time waiting for it).
__host__ __device__ constexpr int epi_warps(int mode) {
  return mode == kModeS2d ? kEpiWarps + kExpWarps : kEpiWarps;
}

template <int kMode>
constexpr int threads_for() {
  return 32 * (kFirstGatherWarp +
               (mode_gathers(kMode) ? producer_warps(kMode) : kTmaProducers - 1));
}


struct SmemCtl {
  // stage s holds K block g (g % kStages == s): its activations (shared
  // memory) and its decoded weights (tensor memory).  full: both operands
  // written; empty: the MMAs that read them have completed.
  uint64_t full[kStages];
  uint64_t empty[kStages];
  uint64_t acc_full[2];     // accumulator b holds a finished tile
  uint64_t acc_empty[2];    // accumulator b has been read by the epilogue
  uint64_t res_full;
  uint64_t mma_drain;      // used only to drain in-flight MMAs after an abort
  uint32_t tmem_base;
  int abort;
  int gtab_off[2][kBK];    // gather: element offset of each code of the K block
  int gtab_rs[2][kBK];     // gather: (r << 16 | s), or -1 beyond the filter
  uint64_t patch_full[2];  // patch mode: a buffer's bulk copy has landed
  uint64_t wready[kMaxResidentKB];   // space-to-depth mode: resident K block decoded
};

constexpr int kSmemLimit = 232448;
constexpr int kPatchMaxKBlocks = 16;   // patch mode keeps a table of every K block's codes

// Dynamic shared memory of a mode: ring, output staging, control block; in
// patch mode also two patch buffers and the code-offset table.
constexpr size_t smem_bytes_for(int mode, size_t patch_cap, int kblocks) {
  return 1024 /*align slack*/ + stages_for(mode) * kStageBytes + kOutStageBytes +
         ((sizeof(SmemCtl) + 15) / 16) * 16 +
         (mode == kModePatch ? 2 * patch_cap + static_cast<size_t>(kblocks) * kBK * 4 : 0);
}
static_assert(smem_bytes_for(kModeTma64, 0, 0) <= kSmemLimit, "shared memory budget");


__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

// 16-bit shared-memory store by 32-bit shared address.
__device__ __forceinline__ void st_shared_u16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(static_cast<uint16_t>(v)) : "memory");
}

struct TileCoord {
  int ktile, q0, p0, n0;
  int split, kb0, kb1;   // K blocks [kb0, kb1) of the filter (split K)
};

__device__ __forceinline__ TileCoord tile_coord(const IgArgs& a, int t) {
  TileCoord c;
  const int d = a.by_base(t);
  c.split = a.cluster ? t - d * a.ksplit : d;
  t = a.cluster ? d : t - d * a.base_tiles;
  c.kb0 = c.split * a.kb_per;
  c.kb1 = min(a.kblocks, c.kb0 + a.kb_per);
  const int pt_lin = a.by_k(t);
  c.ktile = t - pt_lin * a.tiles_k;
  const int np = a.by_tq(pt_lin);
  const int qt = pt_lin - np * a.tiles_q;
  const int nt = a.by_tp(np);
  const int pt = np - nt * a.tiles_p;
  c.q0 = qt * a.bw;
  c.p0 = pt * a.bh;
  c.n0 = nt * a.bn;
  return c;
}

// Direct global store of one output value (the path for fp32 output or
// shapes the TMA store cannot take): fp32 math, residual, ReLU, rounding.
__device__ __forceinline__ float load_residual(const IgArgs& a, size_t o) {
  return a.y_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(a.residual)[o])
                  : static_cast<const float*>(a.residual)[o];
}
__device__ __forceinline__ void store_out(const IgArgs& a, size_t o, float v, float res = 0.0f) {
  if (a.residual) v += res;
  if (a.relu) v = fmaxf(v, 0.0f);
  if (a.y_bf16)
    static_cast<__nv_bfloat16*>(a.y)[o] = __float2bfloat16_rn(v);
  else
    static_cast<float*>(a.y)[o] = v;
}

// Split K in a cluster: its CTAs have stored the sums of one K range each for
// the same tile to a.partial.  Once all have, CTA r adds the ranges of the
// r-th share of the tile's pixels in range order (as splitk_reduce_kernel
// does: the same bits) and applies the epilogue: a warp takes a pixel at a
// time, a lane four filters, all ranges requested at once.  Called by all
// threads; the barrier is reached by every CTA, since every other wait is
// bounded.
__device__ __forceinline__ void add_cluster_sums(const IgArgs& a) {
  cluster_sync();
  const TileCoord tc = tile_coord(a, blockIdx.x);
  const int T = min(a.bn, a.N - tc.n0);   // pixels of the tile: images of a 1 x 1 map
  const int share = (T + a.ksplit - 1) / a.ksplit;
  const int px_end = min(T, share * (tc.split + 1));
  const int k0 = tc.ktile * kBM + 4 * (threadIdx.x & 31);
  if (k0 >= a.K) return;
  const bool vec = (a.K & 3) == 0;   // partial is 16-byte aligned
  const size_t mk = static_cast<size_t>(a.N) * a.K;
  float a2[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) a2[e] = k0 + e < a.K ? 2.0f * __ldg(a.alpha + k0 + e) : 0.0f;
  for (int px = share * tc.split + static_cast<int>(threadIdx.x >> 5); px < px_end;
       px += static_cast<int>(blockDim.x >> 5)) {
    const size_t o = static_cast<size_t>(tc.n0 + px) * a.K + k0;
    float4 v[kMaxCluster];
#pragma unroll
    for (int i = 0; i < kMaxCluster; ++i)
      if (i < a.ksplit) {
        const float* src = a.partial + i * mk + o;
        if (vec) {
          v[i] = __ldcg(reinterpret_cast<const float4*>(src));
        } else {
          v[i].x = __ldcg(src);
          v[i].y = k0 + 1 < a.K ? __ldcg(src + 1) : 0.0f;
          v[i].z = k0 + 2 < a.K ? __ldcg(src + 2) : 0.0f;
          v[i].w = k0 + 3 < a.K ? __ldcg(src + 3) : 0.0f;
        }
      }
    float res[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (a.residual) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (k0 + e < a.K) res[e] = load_residual(a, o + e);
    }
#pragma unroll
    for (int i = 1; i < kMaxCluster; ++i)
      if (i < a.ksplit) {
        v[0].x += v[i].x; v[0].y += v[i].y; v[0].z += v[i].z; v[0].w += v[i].w;
      }
    float y[4] = {a2[0] * v[0].x, a2[1] * v[0].y, a2[2] * v[0].z, a2[3] * v[0].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (a.residual) y[e] += res[e];
      if (a.relu) y[e] = fmaxf(y[e], 0.0f);
    }
    if (vec && a.y_bf16 && (reinterpret_cast<uintptr_t>(a.y) & 7) == 0) {
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(a.y) + o) =
          make_uint2(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]));
    } else if (vec && !a.y_bf16 && (reinterpret_cast<uintptr_t>(a.y) & 15) == 0) {
      *reinterpret_cast<float4*>(static_cast<float*>(a.y) + o) = make_float4(y[0], y[1], y[2], y[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (k0 + e >= a.K) break;
        if (a.y_bf16)
          static_cast<__nv_bfloat16*>(a.y)[o + e] = __float2bfloat16_rn(y[e]);
        else
          static_cast<float*>(a.y)[o + e] = y[e];
      }
    }
  }
}

// Fused quantization prologue: CTA b quantizes filters [b K / G, (b + 1) K / G)
// exactly as the quantize kernel does (the same per-word fields and sums,
// reduced per filter in the same order: bitwise the same codes and alpha),
// with `scratch` (the stage ring, not yet in use) holding a chunk of rows'
// per-word sums and counts; then all CTAs meet at a grid-wide barrier on
// a.gbar (bounded: on expiry the device error word records a timeout and
// the CTA's abort flag is set, so it does no convolution work).
__device__ void quantize_prologue(const IgArgs& a, uint8_t* scratch, int scratch_words,
                                  volatile int* abort_flag) {
  // every thread has read the abort flag before anyone can set it below
  __syncthreads();
  const int G = gridDim.x, b = blockIdx.x, nth = blockDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = static_cast<int>(static_cast<int64_t>(b) * a.K / G);
  const int r1 = static_cast<int>(static_cast<int64_t>(b + 1) * a.K / G);
  const int wpf = a.wpf, n = a.ncodes;
  float* ssum = reinterpret_cast<float*>(scratch);
  int* scnt = reinterpret_cast<int*>(scratch + static_cast<size_t>(scratch_words) * 4);
  const int rows_per_chunk = max(1, scratch_words / wpf);
  for (int c0 = r0; c0 < r1; c0 += rows_per_chunk) {
    const int c1 = min(r1, c0 + rows_per_chunk);
    const int words = (c1 - c0) * wpf;
    // two words per thread per pass: eight 16-byte loads in flight
    for (int i0 = threadIdx.x; i0 < words; i0 += 2 * nth) {
      float v[2][16];
      int nv[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * nth;
        nv[u] = 0;
        if (i < words) {
          const int r = i / wpf, j = i - r * wpf;
          load16(a.wq + static_cast<int64_t>(c0 + r) * n, n, j, a.wq_vec != 0, v[u], nv[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * nth;
        if (i < words) {
          const int r = i / wpf, j = i - r * wpf;
          uint32_t word;
          float sum;
          int c2;
          encode16(v[u], nv[u], word, sum, c2);
          a.codes_w[static_cast<int64_t>(c0 + r) * wpf + j] = word;
          ssum[i] = sum;
          scnt[i] = c2;
        }
      }
    }
    __syncthreads();
    // per filter, as the quantize kernel reduces: words in order by one
    // thread (at most 16 words), else lane-strided and a warp butterfly
    if (wpf <= 16) {
      for (int r = threadIdx.x; r < c1 - c0; r += nth) {
        Sum2 acc{0.0f, 0.0f};
        int cnt2 = 0;
        bool huge = false;
        for (int c = 0; c < wpf; ++c) {
          const float sv = ssum[r * wpf + c];
          huge |= !finite_sum(sv);
          add2(acc, sv);
          cnt2 += scnt[r * wpf + c];
        }
        a.alpha_w[c0 + r] = huge ? alpha_fp64_row(a.wq + static_cast<int64_t>(c0 + r) * n, n)
                                 : alpha_of(acc, cnt2, n);
      }
    } else {
      for (int r = warp; r < c1 - c0; r += nth / 32) {
        Sum2 acc{0.0f, 0.0f};
        int cnt2 = 0;
        bool huge = false;
        for (int c = lane; c < wpf; c += 32) {
          const float sv = ssum[r * wpf + c];
          huge |= !finite_sum(sv);
          add2(acc, sv);
          cnt2 += scnt[r * wpf + c];
        }
        acc = warp_sum2(acc);
        cnt2 = warp_sum(cnt2);
        huge = __any_sync(0xffffffffu, huge);
        if (lane == 0)
          a.alpha_w[c0 + r] = huge ? alpha_fp64_row(a.wq + static_cast<int64_t>(c0 + r) * n, n)
                                   : alpha_of(acc, cnt2, n);
      }
    }
    __syncthreads();
  }
  // grid-wide barrier: every CTA's codes and alpha are written.  A barrier
  // that runs out of time sets the CTA's abort flag (no static shared
  // memory here: the dynamic allocation takes all that the SM offers).
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(a.gbar, 1u);
    const uint64_t t0 = global_timer_ns();
    int ok = 1;
    while (*reinterpret_cast<volatile unsigned*>(a.gbar) < static_cast<unsigned>(G)) {
      if (global_timer_ns() - t0 > kWaitLimitNs) {
        raise_device_error(a.err, TBN_DEVERR_TIMEOUT);
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
    if (!ok) *abort_flag = 1;
  }
  fence_proxy_async_smem();   // the scratch is the ring: TMA writes come after these stores
  __syncthreads();
}

// Place in the K blocks of the tap pairs (kModeTapPair); the last tap of an odd
// number has no partner.
struct TapPairs {
  int m, taps;
  int g, j, na;   // pair, K block within it, 64-channel blocks of the pair
  __device__ __forceinline__ explicit TapPairs(const IgArgs& a)
      : m(a.C / kBK), taps(a.R * a.S), g(0), j(0), na(taps > 1 ? 2 * m : m) {}
  __device__ __forceinline__ bool whole() const { return j < na; }   // a 64-channel block
  __device__ __forceinline__ int second() const { return j >= m ? 1 : 0; }   // of the second tap
  __device__ __forceinline__ void next() {
    if (++j > na) {
      j = 0;
      ++g;
      na = 2 * g + 1 < taps ? 2 * m : m;
    }
  }
};

// kMode: how activations reach the ring (one of the eight kMode... above).
// kPoolBW: 0 = no pool; 8, 16, 32 = fused 2x2/2 max pool for tiles of whole
// output rows of that width; 1 = of any width (a.bw).  kTmaStore: bf16 output
// through the staging tile and TMA stores (else direct global stores).  kFuse:
// with the quantization prologue.
template <int kMode, int kPoolBW, bool kTmaStore, bool kFuse>
__global__ void __launch_bounds__(threads_for<kMode>(), 1)
    conv_igemm_kernel(const __grid_constant__ CUtensorMap tmap_x,
                      const __grid_constant__ CUtensorMap tmap_y,
                      const __grid_constant__ CUtensorMap tmap_res,
                      const __grid_constant__ CUtensorMap tmap_x32,
                      const __grid_constant__ IgArgs a) {
  constexpr bool kGather = mode_gathers(kMode);
  constexpr bool kCh32 = kMode == kModeTma32;
  constexpr bool kPatch = kMode == kModePatch;
  constexpr bool kS2d = kMode == kModeS2d;
  constexpr bool kPad = kMode == kModeTmaPad;
  constexpr bool kRowPair = kMode == kModeRowPair;
  constexpr bool kTapPair = kMode == kModeTapPair;
  constexpr bool kCanCluster = kPoolBW == 0 && !kTmaStore && !kFuse &&
                               (kMode == kModeTma64 || kMode == kModeTma32 || kPad);
  constexpr int kSt = stages_for(kMode);   // ring stages
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned by pointer arithmetic on the shared array, so that the
  // compiler keeps every access derived from it in the shared state space
  uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* ring = smem;                                   // kSt x 32 KiB
  uint8_t* out_stage = smem + kSt * kStageBytes;          // 64 KiB
  SmemCtl* ctl = reinterpret_cast<SmemCtl*>(out_stage + kOutStageBytes);
  // patch mode: two patch buffers, then the code-offset table
  uint8_t* patch_buf = reinterpret_cast<uint8_t*>(ctl) + ((sizeof(SmemCtl) + 15) / 16) * 16;
  volatile int* abort_flag = &ctl->abort;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int KB = a.kblocks;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kSt; ++i) {
      // space-to-depth mode: the weights are resident, only the activation box fills a stage
      mbar_init(&ctl->full[i], (kS2d ? 0 : 32 * kExpWarps) +
                                   (kGather ? 32 * producer_warps(kMode) : 1));
      mbar_init(&ctl->empty[i], 1);
    }
    mbar_init(&ctl->patch_full[0], 1);
    mbar_init(&ctl->patch_full[1], 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl->acc_full[b], 1);
      mbar_init(&ctl->acc_empty[b], 32 * epi_warps(kMode));
    }
    mbar_init(&ctl->res_full, 1);
    mbar_init(&ctl->mma_drain, 1);
    if (kS2d)
      for (int i = 0; i < KB && i < kMaxResidentKB; ++i) mbar_init(&ctl->wready[i], 32 * kExpWarps);
    ctl->abort = 0;
    fence_mbar_init();
    if (!kGather) prefetch_tmap(&tmap_x);
    if (kTapPair) prefetch_tmap(&tmap_x32);
    if (kTmaStore) prefetch_tmap(&tmap_y);
  }
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  if (kS2d) {
    // gather table of the resident K blocks: column j of K block kb (tap
    // (kb / S', kb % S') of the space-to-depth grid, channel j = (dy s + dx)
    // C0 + c) holds original code l = ((s r' + dy) S0 + s s' + dx) C0 + c as
    // (l / 16) | (its magnitude bit) << 16, or ~0 where the s x s block
    // reaches past the filter.  It lives in the output staging tile, which
    // the epilogue first writes after the first tile's MMAs, i.e. after the
    // decode.
    uint32_t* tab = reinterpret_cast<uint32_t*>(out_stage);
    const int ss = a.s2d_s, C0 = a.s2d_C;
    for (int e = threadIdx.x; e < KB * kBK; e += blockDim.x) {
      const int kb = e / kBK, j = e - (e / kBK) * kBK;
      uint32_t v = 0xFFFFFFFFu;
      if (j < ss * ss * C0) {
        const int dy = j / (ss * C0), dx = (j / C0) % ss, c = j % C0;
        const int r = ss * (kb / a.S) + dy, q = ss * (kb % a.S) + dx;
        if (r < a.s2d_R && q < a.s2d_S) {
          const int l = (r * a.s2d_S + q) * C0 + c;
          v = static_cast<uint32_t>(l >> 4) | (static_cast<uint32_t>(code_mag_bit(l & 15)) << 16);
        }
      }
      tab[e] = v;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  // The CTA allocates all 512 columns, so the allocation can only start at
  // lane 0, column 0: every tensor-memory address below is a compile-time
  // constant.  Any other base is reported and the CTA does no work.
  constexpr uint32_t tmem = 0;
  if (ctl->tmem_base != 0u) {
    if (threadIdx.x == 0) {
      raise_device_error(a.err, TBN_DEVERR_BAD_LAUNCH);
      ctl->abort = 1;
    }
  }
  __syncthreads();
  if constexpr (kFuse) {
    if (!*abort_flag)   // uniform: every thread read the flag after the barrier
      quantize_prologue(a, ring, (kSt * kStageBytes) / 8, abort_flag);
  }
  if (*abort_flag) {
    if (warp == 1) tmem_dealloc(ctl->tmem_base, kTmemCols);
    return;   // (the others of a cluster count an exited CTA as arrived)
  }
  const uint32_t acc_tmem = tmem;               // columns [0, 256), or two of 176
  const uint32_t a_tmem0 = tmem + (a.acc2 ? 2u * kAcc2Cols : static_cast<uint32_t>(kAccCols));   // weight ring

  if (!kGather && (warp == 0 || warp >= kFirstGatherWarp)) {
    // ================= TMA producers =================
    grid_dependency_wait();   // activations may come from the previous kernel
    grid_dependents_launch();
    // producer pid issues the K blocks g with g % kTmaProducers == pid; the
    // ring has at least as many stages as producers, so the release a
    // producer waits for always follows the previous release of that slot
    // (the MMA warp releases in order) and its parity wait cannot alias
    const int pid = warp == 0 ? 0 : warp - kFirstGatherWarp + 1;
    int turn = 0;   // g % kTmaProducers
    constexpr int kBoxCh = kCh32 ? kBK / 2 : kBK;   // channels per box
    constexpr int kBoxes = kBK / kBoxCh;             // boxes per K block
    const uint32_t box_bytes = static_cast<uint32_t>(a.bw * a.bh * a.bn * kBoxCh * 2);
    const int cblocks = (a.C + kBoxCh - 1) / kBoxCh;   // boxes per tap
    int g = 0;  // global K-block counter of this CTA
    int st = 0;          // its ring stage
    uint32_t par = 0;    // and the parity of the stage's fill
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
      const TileCoord tc = tile_coord(a, t);
      // base input position of the tile's first pixel
      int w0 = tc.q0 * a.sw - a.pw, h0 = tc.p0 * a.sh - a.ph, n0 = tc.n0;
      if (a.im2col) {
        const int f = tc.p0 * a.Q + tc.q0;
        const int row = a.by_iq(f);
        n0 = a.by_ip(row);
        w0 = (f - row * a.iQ) * a.sw - a.pw;
        h0 = (row - n0 * a.iP) * a.sh - a.ph;
      }
      // (filter row, filter column, channel box) of the next box
      const int tap0 = (tc.kb0 * kBoxes) / cblocks;
      int cb = tc.kb0 * kBoxes - tap0 * cblocks, r = tap0 / a.S, q = tap0 - r * a.S;
      const auto next_box = [&]() {
        if (++cb == cblocks) {
          cb = 0;
          if (++q == a.S) {
            q = 0;
            ++r;
          }
        }
      };
      TapPairs tp(a);   // (r, q): the pair's first tap
      for (int kb = tc.kb0; kb < tc.kb1; ++kb, ++g) {
        const int sb = st;
        const uint32_t ph = par;
        if (++st == kSt) {
          st = 0;
          par ^= 1u;
        }
        const bool mine = turn == pid;
        if (++turn == kTmaProducers) turn = 0;
        if (mine) {
          ok = mbar_wait_warp(&ctl->empty[sb], ph ^ 1u, abort_flag, a.err, kWaitLimitNs);
          if (!ok) break;
          if (kTapPair && elect_one()) {
            mbar_arrive_expect_tx(&ctl->full[sb], box_bytes * kBoxes);
            const bool wrap = q + 1 == a.S;
            const int q1 = wrap ? 0 : q + 1, r1 = wrap ? r + 1 : r;
            const auto box = [&](uint8_t* dst, const CUtensorMap* map, int c0, int dr, int dq) {
              // past the last tap: entirely out of range, it arrives zero-filled
              if (dr >= a.R) {
                c0 = a.C;
                dr = dq = 0;
              }
              if (a.im2col)
                tma_load_im2col_4d(dst, map, &ctl->full[sb], c0, w0, h0, n0, dq, dr);
              else
                tma_load_4d(dst, map, &ctl->full[sb], c0, w0 + dq, h0 + dr, n0);
            };
            uint8_t* dst = ring + sb * kStageBytes;
            if (tp.whole()) {
              const bool s = tp.second();
              box(dst, &tmap_x, kBK * (tp.j - (s ? tp.m : 0)), s ? r1 : r, s ? q1 : q);
            } else {
              box(dst, &tmap_x32, kBK * tp.m, r, q);
              box(dst + kStageBytes / 2, &tmap_x32, kBK * tp.m, r1, q1);
            }
          }
          if (!kTapPair && elect_one()) {
            mbar_arrive_expect_tx(&ctl->full[sb], box_bytes * kBoxes);
            int cb_ = cb, r_ = r, q_ = q;
#pragma unroll
            for (int bx = 0; bx < kBoxes; ++bx) {
              // a box past the filter's last tap is requested at channel C:
              // entirely out of range, it arrives zero-filled
              const bool past = r_ >= a.R;
              uint8_t* dst = ring + sb * kStageBytes + bx * (kStageBytes / kBoxes);
              const int c0 = past ? a.C : cb_ * kBoxCh;
              const int dr = past ? 0 : r_, dq = past ? 0 : q_;
              if (a.im2col)
                tma_load_im2col_4d(dst, &tmap_x, &ctl->full[sb], c0, w0, h0, n0, dq, dr);
              else
                tma_load_4d(dst, &tmap_x, &ctl->full[sb], c0, w0 + dq, h0 + dr, n0);
              if (++cb_ == cblocks) {
                cb_ = 0;
                if (++q_ == a.S) {
                  q_ = 0;
                  ++r_;
                }
              }
            }
          }
          __syncwarp();
        }
        if constexpr (kTapPair) {
          tp.next();
          if (tp.j == 0) {
            q += 2;
            while (q >= a.S) {
              q -= a.S;
              ++r;
            }
          }
        } else {
#pragma unroll
          for (int bx = 0; bx < kBoxes; ++bx) next_box();
        }
      }
    }
    // drain: every copy this warp issued must land before the CTA may exit
    for (int i = g > kSt ? g - kSt : 0; i < g; ++i)
      if (i % kTmaProducers == pid)
        mbar_wait(&ctl->full[i % kSt], static_cast<uint32_t>(i / kSt) & 1u, nullptr,
                  a.err, kWaitLimitNs);
  } else if (kMode == kModeGather && warp >= kFirstGatherWarp) {
    // ================= gather producers =================
    // The gather warps meet at a named barrier every K block, so none of them
    // may leave the loops early: after a failed wait a warp keeps walking the
    // loop structure (reaching every barrier) but does no more work.
    const int gt = threadIdx.x - 32 * kFirstGatherWarp;   // 0..127
    const bool vec = (a.C & 7) == 0;
    grid_dependency_wait();   // activations may come from the previous kernel
    grid_dependents_launch();
    int g = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x) {
      const TileCoord tc = tile_coord(a, t);
      const int T = a.bw * a.bh * a.bn;
      // this thread fills tile rows gt and gt + 128; offset of tap (0, 0)
      int64_t pbase[2];
      int rh[2], rw[2];
      bool rv[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int row = gt + 128 * i;
        const int wi = row % a.bw, hi = (row / a.bw) % a.bh, ni = row / (a.bw * a.bh);
        rh[i] = (tc.p0 + hi) * a.sh - a.ph;
        rw[i] = (tc.q0 + wi) * a.sw - a.pw;
        rv[i] = row < T && tc.n0 + ni < a.N && tc.p0 + hi < a.P && tc.q0 + wi < a.Q;
        pbase[i] = ((static_cast<int64_t>(rv[i] ? tc.n0 + ni : 0) * a.H + rh[i]) * a.W + rw[i]) *
                   static_cast<int64_t>(a.C);
      }
      for (int kb = tc.kb0; kb < tc.kb1; ++kb, ++g) {
        // table of this K block's 64 codes: offset from the tap-(0,0) pixel
        const int tb = g & 1;
        if (gt < kBK) {
          const int k = kb * kBK + gt;
          if (k < a.ncodes) {
            const int c = k % a.C, tap = k / a.C;
            const int r = tap / a.S, s = tap - r * a.S;
            ctl->gtab_off[tb][gt] = (r * a.W + s) * a.C + c;
            ctl->gtab_rs[tb][gt] = (r << 16) | s;
          } else {
            ctl->gtab_off[tb][gt] = 0;
            ctl->gtab_rs[tb][gt] = -1;
          }
        }
        named_barrier_sync(2, 32 * kGatherWarps);
        const int sb = g % kSt;
        const uint32_t it = static_cast<uint32_t>(g / kSt);
        if (ok) ok = mbar_wait(&ctl->empty[sb], (it & 1u) ^ 1u, abort_flag, a.err, kWaitLimitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) continue;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int row = gt + 128 * i;
          if (row >= a.tile_n) continue;
          const uint32_t row_addr = smem_addr(ring + sb * kStageBytes) + static_cast<uint32_t>(row) * 128u;
          uint4 v[8];
          if (vec) {
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
              const int rs = ctl->gtab_rs[tb][ch * 8];
              const int h = rh[i] + (rs >> 16), w = rw[i] + (rs & 0xFFFF);
              v[ch] = make_uint4(0u, 0u, 0u, 0u);
              if (rv[i] && rs >= 0 && h >= 0 && h < a.H && w >= 0 && w < a.W)
                v[ch] = __ldg(reinterpret_cast<const uint4*>(a.x + pbase[i] + ctl->gtab_off[tb][ch * 8]));
            }
          } else {
            const unsigned short* xs = reinterpret_cast<const unsigned short*>(a.x);
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
              uint32_t e[8];
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int rs = ctl->gtab_rs[tb][ch * 8 + q];
                const int h = rh[i] + (rs >> 16), w = rw[i] + (rs & 0xFFFF);
                e[q] = 0u;
                if (rv[i] && rs >= 0 && h >= 0 && h < a.H && w >= 0 && w < a.W)
                  e[q] = __ldg(xs + pbase[i] + ctl->gtab_off[tb][ch * 8 + q]);
              }
              v[ch] = make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16),
                                 e[6] | (e[7] << 16));
            }
          }
#pragma unroll
          for (int ch = 0; ch < 8; ++ch)  // 128-byte swizzle: chunk XOR (row mod 8)
            st_shared_v4(row_addr + static_cast<uint32_t>(((ch ^ (row & 7)) & 7) * 16), v[ch]);
        }
        fence_proxy_async_smem();   // generic-proxy writes -> visible to tcgen05.mma
        mbar_arrive(&ctl->full[sb]);
      }
    }
  } else if (kPatch && warp >= kFirstGatherWarp) {
    // ================= patch producers =================
    // Tiles are whole output rows of one image (bn = 1, tiles_q = 1).  The
    // input rows a tile reads, [p0 sh - ph, + PR) x [-pw, W + pw) x C, are
    // staged in a shared-memory patch (zero outside the image); each K block
    // row is then built from the patch with one 32-bit load per pair of codes
    // when the pair is contiguous there, two 16-bit loads otherwise.  With no
    // column padding the in-image rows are one contiguous range of x and one
    // bulk copy (issued a tile ahead, into the other buffer) fetches them.
    const int gt = threadIdx.x - 32 * kFirstGatherWarp;   // 0..255
    const int pitch = a.PW * a.C;                          // patch row, elements
    const int patch_elems = a.PR * pitch;
    const int* ptab = reinterpret_cast<const int*>(patch_buf + 2 * a.patch_cap);
    int* ptab_w = reinterpret_cast<int*>(patch_buf + 2 * a.patch_cap);
    const uint8_t* xb = reinterpret_cast<const uint8_t*>(a.x);
    // offset table of every K block: patch element of code k relative to the
    // pixel's (tap 0, channel 0) element, -1 past the filter
    for (int i = gt; i < KB * kBK; i += 32 * kPatchWarps) {
      const int k = i;
      int off = -1;
      if (k < a.ncodes) {
        const int c = k % a.C, tap = k / a.C;
        const int r = tap / a.S, s = tap - r * a.S;
        off = (r * a.PW + s) * a.C + c;
      }
      asm volatile("st.shared.s32 [%0], %1;" ::"r"(smem_addr(ptab_w + i)), "r"(off) : "memory");
    }
    grid_dependency_wait();   // activations may come from the previous kernel
    grid_dependents_launch();
    named_barrier_sync(2, 32 * kPatchWarps);

    // geometry of tile t's patch: in-image patch rows [lo, hi), the byte
    // offset `src` in x of its first in-image element, and the byte offset of
    // patch element 0 in its buffer (chosen so that the bulk copy's
    // destination is 16-byte aligned)
    auto geom = [&](int t, int& lo, int& hi, long long& src, uint32_t& off0) {
      const TileCoord tc = tile_coord(a, t);
      const int h0 = tc.p0 * a.sh - a.ph;
      lo = max(0, -h0);
      hi = min(a.PR, a.H - h0);
      if (hi < lo) hi = lo;
      const long long e0 = static_cast<long long>(lo) * pitch;
      src = ((static_cast<long long>(tc.n0) * a.H + h0 + lo) * a.W) * a.C * 2;
      off0 = static_cast<uint32_t>(((src & 15) - 2 * e0) & 15);
    };
    // one thread: the bulk copy of tile t's in-image rows into buffer b
    auto issue = [&](int t, int b) {
      int lo, hi;
      long long src;
      uint32_t off0;
      geom(t, lo, hi, src, off0);
      const long long len = static_cast<long long>(hi - lo) * pitch * 2;
      const long long a0 = src & ~15LL;
      long long a1 = (src + len + 15) & ~15LL;
      if (a1 > a.x_bytes) a1 = a.x_bytes & ~15LL;   // the rest is copied by threads
      const uint32_t bytes = a1 > a0 ? static_cast<uint32_t>(a1 - a0) : 0u;
      uint8_t* dst = patch_buf + b * a.patch_cap + off0 + 2 * static_cast<long long>(lo) * pitch -
                     (src & 15);
      fence_proxy_async_smem();   // earlier generic accesses of the buffer come first
      mbar_arrive_expect_tx(&ctl->patch_full[b], bytes);
      if (bytes) bulk_load_1d(dst, xb + a0, bytes, &ctl->patch_full[b]);
    };

    int g = 0;
    bool ok = true;
    uint32_t issued[2] = {0u, 0u};   // bulk copies issued into each buffer (thread 0)
    uint32_t landed[2] = {0u, 0u};   // copies this thread has seen complete
    uint32_t tiles_done = 0;
    if (a.patch_bulk && gt == 0 && static_cast<int>(blockIdx.x) < a.tiles) {
      issue(blockIdx.x, 0);
      ++issued[0];
    }
    __syncwarp();   // reconverge before the aligned named barriers below
    const int T = a.bw * a.bh;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++tiles_done) {
      const TileCoord tc = tile_coord(a, t);
      const int b = tiles_done & 1;
      uint8_t* buf = patch_buf + b * a.patch_cap;
      int lo, hi;
      long long src;
      uint32_t off0;
      geom(t, lo, hi, src, off0);
      const uint32_t buf_s = smem_addr(buf);
      const uint32_t pe_s = buf_s + off0;   // patch element e at pe_s + 2 e
      // everyone has finished building the previous tile (the buffer filled
      // next was last read two tiles ago)
      named_barrier_sync(2, 32 * kPatchWarps);
      if (a.patch_bulk) {
        if (gt == 0 && ok && t + static_cast<int>(gridDim.x) < a.tiles) {
          issue(t + gridDim.x, b ^ 1);
          ++issued[b ^ 1];
        }
        if (ok) {
          ok = mbar_wait(&ctl->patch_full[b], landed[b] & 1u, abort_flag, a.err, kWaitLimitNs);
          if (ok) ++landed[b];
        }
        ok = __all_sync(0xffffffffu, ok);
        // rows outside the image are zero; the copy's rounding may have
        // written neighbouring bytes there
        for (int e = gt; e < lo * pitch; e += 32 * kPatchWarps) st_shared_u16(pe_s + 2 * e, 0u);
        for (int e = hi * pitch + gt; e < patch_elems; e += 32 * kPatchWarps)
          st_shared_u16(pe_s + 2 * e, 0u);
        // the last bytes of x that no 16-byte chunk of the copy covered
        const long long len = static_cast<long long>(hi - lo) * pitch * 2;
        const long long cov = a.x_bytes & ~15LL;
        if (src + len > cov) {
          const long long first = max(src, cov);
          for (long long bpos = first + 2 * gt; bpos < src + len; bpos += 2 * 32 * kPatchWarps)
            st_shared_u16(pe_s + 2 * static_cast<uint32_t>(lo * pitch + (bpos - src) / 2),
                          *reinterpret_cast<const uint16_t*>(xb + bpos));
        }
      } else {
        // column padding: element by element, zero outside the image
        const TileCoord tc = tile_coord(a, t);
        const int h0 = tc.p0 * a.sh - a.ph;
        const uint16_t* xs = reinterpret_cast<const uint16_t*>(a.x);
        for (int e = gt; e < patch_elems; e += 32 * kPatchWarps) {
          const int rho = e / pitch, rem = e - rho * pitch;
          const int u = rem / a.C, c = rem - u * a.C;
          const int h = h0 + rho, w = u - a.pw;
          uint16_t v = 0;
          if (h >= 0 && h < a.H && w >= 0 && w < a.W)
            v = __ldg(xs + ((static_cast<long long>(tc.n0) * a.H + h) * a.W + w) * a.C + c);
          st_shared_u16(pe_s + 2 * e, v);
        }
      }
      named_barrier_sync(2, 32 * kPatchWarps);   // patch complete
      // this thread's rows: pixel (i, q) of the tile reads from patch element
      // i sh pitch + q sw C on; base in 16-bit units from the buffer start
      constexpr int kRows = kMaxTileN / (32 * kPatchWarps);   // operand rows per thread
      int base[kRows];
      bool valid[kRows];
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const int px = gt + 32 * kPatchWarps * j;
        const int i = px / a.bw, q = px - i * a.bw;
        valid[j] = px < T;
        base[j] = static_cast<int>(off0 / 2) + i * a.sh * pitch + q * a.sw * a.C;
      }
      for (int kb = tc.kb0; kb < tc.kb1; ++kb, ++g) {
        const int sb = g % kSt;
        const uint32_t it = static_cast<uint32_t>(g / kSt);
        if (ok) ok = mbar_wait(&ctl->empty[sb], (it & 1u) ^ 1u, abort_flag, a.err, kWaitLimitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) continue;
        const int* __restrict__ tab = ptab + kb * kBK;
        uint8_t* __restrict__ stage = ring + sb * kStageBytes;
        const uint16_t* __restrict__ p16 = reinterpret_cast<const uint16_t*>(buf);
        const uint32_t* __restrict__ p32 = reinterpret_cast<const uint32_t*>(buf);
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
          const int row = gt + 32 * kPatchWarps * j;
          if (row >= a.tile_n) continue;
          // four chunks at a time: every load of the group is issued before
          // the first shift or store
#pragma unroll
          for (int cg = 0; cg < 2; ++cg) {
            int4 o[8];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              o[2 * c] = *reinterpret_cast<const int4*>(tab + 8 * (4 * cg + c));
              o[2 * c + 1] = *reinterpret_cast<const int4*>(tab + 8 * (4 * cg + c) + 4);
            }
            uint32_t wv[4][5];
            bool run[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              // the chunk's 8 codes are 8 consecutive patch elements (one run
              // of a filter row): 5 aligned words, 4 funnel shifts
              run[c] = valid[j] && o[2 * c].x >= 0 && o[2 * c + 1].w == o[2 * c].x + 7;
              const int e = base[j] + (o[2 * c].x >= 0 ? o[2 * c].x : 0);
              const uint32_t* w = p32 + (e >> 1);
#pragma unroll
              for (int u = 0; u < 5; ++u) wv[c][u] = run[c] ? w[u] : 0u;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int ch = 4 * cg + c;
              uint4 v = make_uint4(0u, 0u, 0u, 0u);
              if (run[c]) {
                const int e = base[j] + o[2 * c].x;
                const uint32_t sh = static_cast<uint32_t>(e & 1) * 16u;
                v.x = __funnelshift_r(wv[c][0], wv[c][1], sh);
                v.y = __funnelshift_r(wv[c][1], wv[c][2], sh);
                v.z = __funnelshift_r(wv[c][2], wv[c][3], sh);
                v.w = __funnelshift_r(wv[c][3], wv[c][4], sh);
              } else if (valid[j]) {
                // a chunk across two filter rows, or past the filter's end
                const int off[8] = {o[2 * c].x, o[2 * c].y, o[2 * c].z, o[2 * c].w,
                                    o[2 * c + 1].x, o[2 * c + 1].y, o[2 * c + 1].z,
                                    o[2 * c + 1].w};
                uint32_t h[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                  h[u] = off[u] >= 0 ? static_cast<uint32_t>(p16[base[j] + off[u]]) : 0u;
                v = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16),
                               h[6] | (h[7] << 16));
              }
              // 128-byte swizzle: chunk XOR (row mod 8)
              *reinterpret_cast<uint4*>(stage + row * 128 + (((ch ^ (row & 7)) & 7) << 4)) = v;
            }
          }
        }
        fence_proxy_async_smem();   // generic-proxy writes -> visible to tcgen05.mma
        mbar_arrive(&ctl->full[sb]);
      }
    }
    // drain (after an abort): every bulk copy issued must land before the
    // CTA may exit
    if (a.patch_bulk && gt == 0) {
      for (int b = 0; b < 2; ++b)
        while (landed[b] < issued[b] &&
               mbar_wait(&ctl->patch_full[b], landed[b] & 1u, nullptr, a.err, kWaitLimitNs))
          ++landed[b];
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================= MMA issuer =================
    const uint32_t idesc = idesc_bf16_f32(kBM, static_cast<uint32_t>(a.tile_n));
    int issued = 0, st = 0;
    uint32_t tiles_done = 0, par = 0;
    const int tap_blocks = (a.C + kBK - 1) / kBK;   // padded mode: K blocks per tap
    const int tap_row = a.S * (a.C / kBK);          // row pairs: K blocks per tap row
    // space-to-depth mode: K steps that hold channels (the others are zero in
    // both operands; AlexNet conv1, batch 256, three of four: 83.8 -> 79.4 us)
    const int s2d_steps = (a.s2d_s * a.s2d_s * a.s2d_C + 15) / 16;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++tiles_done) {
      const TileCoord tc = tile_coord(a, t);
      // the epilogue must have drained this accumulator's previous tile
      const uint32_t ab = a.acc2 ? (tiles_done & 1u) : 0u;
      const uint32_t use = a.acc2 ? (tiles_done >> 1) : tiles_done;   // uses of accumulator ab
      const uint32_t acc_t = acc_tmem + ab * kAcc2Cols;
      ok = mbar_wait_warp(&ctl->acc_empty[ab], (use & 1u) ^ 1u, abort_flag, a.err, kWaitLimitNs);
      if (!ok) break;
      TapPairs tp(a);
      int left = kPad ? a.C - kBK * (tc.kb0 % tap_blocks) : kBK;   // channels left in the tap
      for (int kb = tc.kb0; kb < tc.kb1; ++kb) {
        ok = mbar_wait_warp(&ctl->full[st], par, abort_flag, a.err, kWaitLimitNs);
        if (kS2d && tiles_done == 0 && ok)   // first use of a resident K block
          ok = mbar_wait_warp(&ctl->wready[kb], 0u, abort_flag, a.err, kWaitLimitNs);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t a_col =
            kS2d ? static_cast<uint32_t>(kTmemCols - 8 * s2d_steps * (KB - kb))
                 : a_tmem0 + static_cast<uint32_t>(st * kAColsPerStage);
        // K step kk: 16 codes = 8 TMEM columns of A, 32 bytes of B rows (two
        // halves of 32 codes, 64-byte rows, with 32-channel boxes)
        const uint32_t b_addr = smem_addr(ring) + static_cast<uint32_t>(st * kStageBytes);
        constexpr uint32_t kHalf = kCh32 ? (kStageBytes / 2) >> 4 : 4u;
        // row pairs: the first tap row's blocks are the lower half's alone, the
        // last one's the upper half's
        if (kRowPair && (kb <= tap_row || kb >= KB - tap_row))
          tc_mma_ts_block_halves(acc_t, a_col, smem_desc_sw128_kmajor(b_addr), idesc,
                                 kb != 0 ? 1u : 0u, kb >= KB - tap_row ? ~0u : 0u,
                                 kb <= tap_row ? ~0u : 0u, kb < tap_row ? ~0u : 0u,
                                 &ctl->empty[st], kb == KB - 1 ? &ctl->acc_full[ab] : nullptr);
        else if (kTapPair && !tp.whole())
          tc_mma_ts_block<2, (kStageBytes / 2 >> 4), (kStageBytes / 2 >> 4) + 2>(
              acc_t, a_col, smem_desc_sw64_kmajor(b_addr), idesc, kb != tc.kb0 ? 1u : 0u, 4,
              &ctl->empty[st], kb == tc.kb1 - 1 ? &ctl->acc_full[ab] : nullptr);
        else tc_mma_ts_block<2, kHalf, kHalf + 2>(
            acc_t, a_col, kCh32 ? smem_desc_sw64_kmajor(b_addr) : smem_desc_sw128_kmajor(b_addr),
            idesc, kb != tc.kb0 ? 1u : 0u, kPad ? (left + 15) / 16 : kS2d ? s2d_steps : 4, &ctl->empty[st],
            kb == tc.kb1 - 1 ? &ctl->acc_full[ab] : nullptr);
        if (kPad) left = left > kBK ? left - kBK : a.C;
        if (kTapPair) tp.next();
        ++issued;
        if (++st == kSt) {
          st = 0;
          par ^= 1u;
        }
      }
    }
    if (!ok && issued > 0) {
      // drain in-flight MMAs before TMEM is freed
      if (elect_one()) tc_commit(&ctl->mma_drain);
      __syncwarp();
      mbar_wait(&ctl->mma_drain, 0u, nullptr, a.err, kWaitLimitNs);
    }
  } else if (warp >= kFirstExpWarp && warp < kFirstExpWarp + kExpWarps) {
    // ================= expanders =================
    const int sub = warp & 3;                         // TMEM sub-partition
    const int half = (warp - kFirstExpWarp) >> 2;     // which 32 codes of a K block
    const int m = sub * 32 + lane;                    // filter row within the tile
    const uint32_t lane_off = static_cast<uint32_t>(sub * 32) << 16;
    if constexpr (kS2d) {
      // Decode every K block of the filter once into its resident columns,
      // the last of which end at 512: eight for each K step that holds
      // channels (this warp: those of codes [32 half, + 32)).  Filter rows
      // past K hold zeros.
      const uint32_t* tab = reinterpret_cast<const uint32_t*>(out_stage);
      const uint32_t* crow = m < a.K ? a.codes + static_cast<size_t>(m) * a.wpf : nullptr;
      const int cols = 8 * ((a.s2d_s * a.s2d_s * a.s2d_C + 15) / 16);
      const int part = min(16, cols - 16 * half);   // 16, 8 or none
      grid_dependency_wait();   // the codes may come from the previous kernel
      for (int kb = 0; kb < KB; ++kb) {
        uint32_t v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const uint32_t e0 = tab[kb * kBK + 32 * half + 2 * i];
          const uint32_t e1 = tab[kb * kBK + 32 * half + 2 * i + 1];
          uint32_t lo = 0u, hi = 0u;
          // W~/2 in bf16: 0x3F00 (0.5) | m << 7 (1.0) | s << 15
          if (crow != nullptr && e0 != 0xFFFFFFFFu)
            lo = ((__ldg(crow + (e0 & 0xFFFFu)) >> (e0 >> 16)) & 0x101u) * 128u + 0x3F00u;
          if (crow != nullptr && e1 != 0xFFFFFFFFu)
            hi = ((__ldg(crow + (e1 & 0xFFFFu)) >> (e1 >> 16)) & 0x101u) * 128u + 0x3F00u;
          v[i] = lo | (hi << 16);
        }
        const uint32_t col =
            tmem + lane_off + static_cast<uint32_t>(kTmemCols - cols * (KB - kb) + 16 * half);
        if (part == 16) tmem_st_32x32b_x16(col, v);
        else if (part == 8) tmem_st_32x32b_x8(col, v);
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(&ctl->wready[kb]);
      }
    } else {
    const bool pair_ok = ((a.wpf & 1) == 0) && ((reinterpret_cast<uintptr_t>(a.codes) & 7) == 0);
    // this CTA's K blocks, all tiles in sequence
    int total = 0;
    if (a.ksplit == 1) {
      total = (a.tiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) /
              static_cast<int>(gridDim.x) * KB;
    } else {
      for (int t = blockIdx.x; t < a.tiles; t += gridDim.x) {
        const TileCoord tc = tile_coord(a, t);
        total += tc.kb1 - tc.kb0;
      }
    }
    // prefetch cursor over (tile, kb): the codes of K block kb of a filter
    // are words [4 kb, 4 kb + 4) of its row; this warp takes two of them,
    // where the row has them (kb < kb_lim)
    int t_ld = blockIdx.x, kb_ld = 0, kb_end = 0, kb_lim = 0;
    const int kb_words = (a.wpf - 2 * half + 3) / 4;   // K blocks whose two words begin in the row
    // row pairs: the upper 64 rows (two of the four sub-partitions) run one
    // tap row behind; what is stored in the K blocks before and after a half's
    // taps is of no account (the MMA leaves that half's accumulators alone)
    const int behind = kRowPair && sub >= 2 ? a.S * (a.C / kBK) : 0;
    const int kb_taps = kRowPair ? (a.R - 1) * a.S * (a.C / kBK) : 0;
    const uint32_t* cp = a.codes;
    // padded mode: this half block's first code, and channels left in its tap
    const int tap_blocks = (a.C + kBK - 1) / kBK;
    int code0 = 0, ch_left = 0;
    TapPairs tp(a);
    auto set_row = [&]() {
      const TileCoord tc = tile_coord(a, t_ld < a.tiles ? t_ld : 0);
      kb_ld = tc.kb0;
      kb_end = tc.kb1;
      const int k = kRowPair ? (m & 63) : tc.ktile * kBM + m;
      const bool in = t_ld < a.tiles && k < a.K;
      if constexpr (kRowPair) {
        kb_lim = in ? kb_taps : 0;
        kb_ld = -behind;
        kb_end = KB - behind;
        cp = a.codes + static_cast<int64_t>(in ? k : 0) * a.wpf + 4 * kb_ld + 2 * half;
        return;
      }
      if constexpr (kPad) {
        const int tap = kb_ld / tap_blocks, cb = kb_ld - tap * tap_blocks;
        ch_left = a.C - kBK * cb;
        code0 = tap * a.C + kBK * cb + 32 * half;
        kb_lim = in ? kb_end : 0;
        cp = a.codes + static_cast<size_t>(in ? k : 0) * a.wpf;
        return;
      }
      if constexpr (kTapPair) {
        tp = TapPairs(a);
        kb_lim = in ? kb_end : 0;
        cp = a.codes + static_cast<size_t>(in ? k : 0) * a.wpf;
        return;
      }
      kb_lim = in ? kb_words : 0;
      cp = a.codes + static_cast<size_t>(in ? k : 0) * a.wpf + 4 * kb_ld + 2 * half;
    };
    set_row();
    // the two words of a half K block; in padded mode the three words that hold
    // its codes and whether they begin in the middle of the first, put together
    // when they are decoded: put together here, every K block would wait for
    // its own loads (27 x 27, 56 channels, 5 x 5, 128 filters, batch 32: 13.5 us
    // so, 12.1 now)
    struct Codes {
      uint32_t x, y, z;
      bool mid;
    };
    const auto decode = [&](const Codes& q, uint32_t* v, const PairMultipliers& pm) {
      uint32_t x = q.x, y = q.y;
      if (kPad && q.mid) {
        x = ((x >> 4) & 0x0F0F0F0Fu) | ((y & 0x0F0F0F0Fu) << 4);
        y = ((y >> 4) & 0x0F0F0F0Fu) | ((q.z & 0x0F0F0F0Fu) << 4);
      }
      word_to_bf16x2(x, v, pm);
      word_to_bf16x2(y, v + 8, pm);
    };
    auto next_codes = [&]() -> Codes {
      Codes r{0u, 0u, 0u, false};
      if constexpr (kPad) {
        // 32 codes from code0 on (a multiple of 8: whole words, or the upper
        // half of one and the lower half of the next), fewer where the tap
        // ends: other columns multiply zero activations
        const int n = min(32, ch_left - 32 * half);
        if (kb_ld < kb_lim && n > 0) {
          const int w = code0 >> 4, end = (code0 & 8) + n;
          r.mid = (code0 & 8) != 0;
          r.x = __ldg(cp + w);
          if (end > 16) r.y = __ldg(cp + w + 1);
          if (end > 32) r.z = __ldg(cp + w + 2);
        }
        if (ch_left > kBK) {
          ch_left -= kBK;
          code0 += kBK;
        } else {
          code0 += ch_left;
          ch_left = a.C;
        }
        if (++kb_ld == kb_end) {
          t_ld += gridDim.x;
          set_row();
        }
        return r;
      }
      // tap pairs: the words of the block's tap (4 m + 2 each)
      const uint32_t* wp = cp;
      bool there = true;
      if constexpr (kTapPair) {
        const bool w = tp.whole();
        const int s = w ? tp.second() : half;
        wp += (2 * tp.g + s) * (4 * tp.m + 2) + 4 * (w ? tp.j - (s ? tp.m : 0) : tp.m) +
              (w ? 2 * half : 0);
        there = 2 * tp.g + s < tp.taps;
        tp.next();
      }
      if (there && kb_ld < kb_lim && (!kRowPair || kb_ld >= 0)) {
        // written by this launch's prologue when fused: ordinary (L1-cached,
        // coherent) loads after the grid barrier's acquire then, not the
        // read-only path, which assumes data constant for the whole launch
        const bool two = kTapPair || 4 * kb_ld + 2 * half + 1 < a.wpf;
        uint2 t;
        if constexpr (kFuse) {
          if (pair_ok) t = __ldca(reinterpret_cast<const uint2*>(wp));
          else t = make_uint2(__ldca(wp), two ? __ldca(wp + 1) : 0u);
        } else {
          if (pair_ok) t = __ldg(reinterpret_cast<const uint2*>(wp));
          else t = make_uint2(__ldg(wp), two ? __ldg(wp + 1) : 0u);
        }
        r.x = t.x;
        r.y = t.y;
      }
      if constexpr (!kTapPair) cp += 4;
      if (++kb_ld == kb_end) {
        t_ld += gridDim.x;
        set_row();
      }
      return r;
    };
    const PairMultipliers pm;
    grid_dependency_wait();   // the codes may come from the previous kernel
    Codes q0 = next_codes(), q1 = next_codes(), q2 = next_codes(), q3 = next_codes();
    const uint32_t col = a_tmem0 + lane_off + static_cast<uint32_t>(16 * half);
    // two K blocks per iteration: their tensor-memory stores share one
    // tcgen05.wait::st
    int st = 0;         // ring stage of the next K block
    uint32_t par = 0;   // parity of its fill
    for (int g = 0; g < total; g += 2) {
      const bool two = g + 1 < total;   // warp-uniform
      uint32_t v0[16], v1[16];
      decode(q0, v0, pm);
      decode(q1, v1, pm);
      q0 = q2;
      q1 = q3;
      q2 = next_codes();
      q3 = next_codes();
      const int s0 = st;
      const uint32_t p0 = par ^ 1u;
      if (++st == kSt) { st = 0; par ^= 1u; }
      const int s1 = st;
      const uint32_t p1 = par ^ 1u;
      if (++st == kSt) { st = 0; par ^= 1u; }
      // in patch mode the operand builders are the bottleneck: waiting
      // expanders park instead of spinning, leaving the issue slots to them
      bool ok = kPatch ? mbar_wait_sleep(&ctl->empty[s0], p0, abort_flag, a.err, kWaitLimitNs)
                       : mbar_wait(&ctl->empty[s0], p0, abort_flag, a.err, kWaitLimitNs);
      if (ok && two)
        ok = kPatch ? mbar_wait_sleep(&ctl->empty[s1], p1, abort_flag, a.err, kWaitLimitNs)
                    : mbar_wait(&ctl->empty[s1], p1, abort_flag, a.err, kWaitLimitNs);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      tmem_st_32x32b_x16(col + static_cast<uint32_t>(s0 * kAColsPerStage), v0);
      if (two) tmem_st_32x32b_x16(col + static_cast<uint32_t>(s1 * kAColsPerStage), v1);
      tmem_wait_st();
      tc_fence_before_sync();
      mbar_arrive(&ctl->full[s0]);
      if (two) mbar_arrive(&ctl->full[s1]);
    }
    }
  }
  if ((warp >= kFirstEpiWarp && warp < kFirstEpiWarp + kEpiWarps) ||
      (kS2d && warp >= kFirstExpWarp && warp < kFirstExpWarp + kExpWarps)) {
    // ================= epilogue =================
    // kParts warps per TMEM sub-partition, each reading a part of the columns.
    constexpr int kParts = epi_warps(kMode) / 4;
    const int sub = warp & 3;
    const int half = warp >= kFirstEpiWarp ? (warp - kFirstEpiWarp) >> 2
                                           : kEpiWarps / 4 + ((warp - kFirstExpWarp) >> 2);
    const int m = sub * 32 + lane;
    const bool elected = threadIdx.x == 32 * kFirstEpiWarp;
    const uint32_t lane_off = static_cast<uint32_t>(sub * 32) << 16;
    const int Po = kPoolBW ? a.P / 2 : a.P;
    const int Qo = kPoolBW ? a.Q / 2 : a.Q;
    const uint32_t res_half_bytes = static_cast<uint32_t>(a.bw * a.bh * a.bn * (kBM / 2) * 2);
    __nv_bfloat16* stage = reinterpret_cast<__nv_bfloat16*>(out_stage);
    grid_dependency_wait();   // the residual may come from the previous kernel
    uint32_t tiles_done = 0;
    bool ok = true;
    // The epilogue warps meet at named barriers, so after a failed wait they
    // keep walking the tile loop (reaching every barrier) without working.
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++tiles_done) {
      const TileCoord tc = tile_coord(a, t);
      const uint32_t par = tiles_done & 1u;   // the residual box
      const uint32_t ab = a.acc2 ? (tiles_done & 1u) : 0u;
      const uint32_t apar = (a.acc2 ? (tiles_done >> 1) : tiles_done) & 1u;
      const uint32_t acc_b = acc_tmem + ab * kAcc2Cols;
      const uint32_t acc = acc_b + lane_off;
      const int k = kRowPair ? (m & 63) : tc.ktile * kBM + m;
      const bool kvalid = k < a.K;
      const float a2 = kvalid ? 2.0f * (kFuse ? __ldca(a.alpha + k) : __ldg(a.alpha + k)) : 0.0f;
      // fragment epilogue: 2 alpha, twice, of this lane's filters (requested
      // before the accumulator is waited for)
      const int fr = lane >> 2;   // fragment row within 8
      uint64_t a2f[2][2];
      if constexpr (kPoolBW == 0 && kTmaStore) {
#pragma unroll
        for (int lg = 0; lg < 2; ++lg) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int mm = sub * 32 + lg * 16 + u * 8 + fr;
            const int kk = kRowPair ? (mm & 63) : tc.ktile * kBM + mm;
            const float s2 =
                kk < a.K ? 2.0f * (kFuse ? __ldca(a.alpha + kk) : __ldg(a.alpha + kk)) : 0.0f;
            a2f[lg][u] = f32x2(__float_as_uint(s2), __float_as_uint(s2));
          }
        }
      }
      if (kTmaStore) {
        // the previous tile's store must have finished reading the staging tile
        if (elected) bulk_wait_group_read<0>();
        named_barrier_sync(1, 32 * epi_warps(kMode));
        if (ok && a.residual && elected) {
          // the residual box, in the staging tile's own layout (two swizzled
          // halves of 64 filters), lands where the outputs will be staged
          const bool both = kRowPair || tc.ktile * kBM + kBM / 2 < a.K;
          mbar_arrive_expect_tx(&ctl->res_full, both ? 2 * res_half_bytes : res_half_bytes);
          if constexpr (kRowPair) {   // (filter, column, row parity, row pair)
            tma_load_4d(stage, &tmap_res, &ctl->res_full, 0, 0, 0, tc.p0);
            tma_load_4d(reinterpret_cast<uint8_t*>(stage) + 32768, &tmap_res, &ctl->res_full, 0, 0,
                        1, tc.p0);
          } else {
            tma_load_4d(stage, &tmap_res, &ctl->res_full, tc.ktile * kBM, tc.q0, tc.p0, tc.n0);
          }
          if (!kRowPair && both)
            tma_load_4d(reinterpret_cast<uint8_t*>(stage) + 32768, &tmap_res, &ctl->res_full,
                        tc.ktile * kBM + kBM / 2, tc.q0, tc.p0, tc.n0);
        }
      }
      if (ok)
        ok = kPatch ? mbar_wait_sleep(&ctl->acc_full[ab], apar, abort_flag, a.err, kWaitLimitNs)
                    : mbar_wait(&ctl->acc_full[ab], apar, abort_flag, a.err, kWaitLimitNs);
      if (kTmaStore && a.residual && ok)
        ok = mbar_wait(&ctl->res_full, par, abort_flag, a.err, kWaitLimitNs);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) tc_fence_after_sync();
      if (!ok) {
        // skip the work, keep the barrier schedule
      } else if constexpr (kPoolBW == 0 && kTmaStore) {
        // Fragment epilogue: 16x256b loads (lane = filter, column = pixel),
        // scale / residual / ReLU / bf16 pairs, transposed 8x8 stores into
        // the staging tile [pixel][filter] as two 128-byte-swizzled halves of
        // 64 filters (chunk c of pixel row px at c ^ (px & 7)).  The residual
        // sits at the very addresses its outputs go to, and the transposed
        // 8x8 loads deliver it in the fragment's own register layout, so it
        // costs one ldmatrix per stmatrix.  (One 2-byte shared load and store
        // per value took a 64-filter 56x56 layer at batch 128 from 49 to
        // 103 us; this way the residual costs 51.4 MB more of reads, no more.)
        const int nchunks = (a.tile_n + 31) / 32;
        const int c_begin = (nchunks * half + kParts - 1) / kParts;
        const int c_end = (nchunks * (half + 1) + kParts - 1) / kParts;
        // this lane's stmatrix row address pieces: matrix mi = lane / 8, row = lane % 8
        const int mi = lane >> 3, mrow = lane & 7;
        const uint32_t stage_s = smem_addr(stage);
        // 16 lanes (filters) at a time: the other 16 lanes' columns are on
        // their way while these are processed.  The accumulator is released
        // once the last have arrived.
        uint32_t v[2][16];
        const auto load = [&](int j, int lg) {
          tmem_ld_16x256b_x4(acc_b + (static_cast<uint32_t>(sub * 32 + lg * 16) << 16) +
                                 static_cast<uint32_t>(32 * j),
                             v[lg]);
        };
        if (c_begin < c_end) load(c_begin, 0);
        for (int j = c_begin; j < c_end; ++j) {
#pragma unroll
          for (int lg = 0; lg < 2; ++lg) {
            tmem_wait_ld();
            if (lg == 0) {
              load(j, 1);
            } else if (j + 1 < c_end) {
              load(j + 1, 0);
            } else {
              tc_fence_before_sync();
              mbar_arrive(&ctl->acc_empty[ab]);
            }
            uint32_t pk[8];
            uint32_t addr[2];
#pragma unroll
            for (int bp = 0; bp < 2; ++bp) {
              // matrices: (filters +0, block 2bp), (+8, 2bp), (+0, 2bp+1), (+8, 2bp+1)
              const int px = 32 * j + 8 * (2 * bp + (mi >> 1)) + mrow;
              const int chunk = 4 * sub + 2 * lg + (mi & 1);           // 8-filter chunk 0..15
              addr[bp] = stage_s + static_cast<uint32_t>((chunk >> 3) * 32768 + px * 128 +
                                                         (((chunk & 7) ^ (px & 7)) << 4));
            }
            if (a.residual) {
#pragma unroll
              for (int bp = 0; bp < 2; ++bp)
                ldmatrix_x4_trans(addr[bp], pk[4 * bp + 0], pk[4 * bp + 1], pk[4 * bp + 2],
                                  pk[4 * bp + 3]);
            }
            // pk[2b], pk[2b + 1]: pixels 2 (lane % 4) + 0/1 of block b, filters fr
            // and fr + 8
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const uint64_t acc2x = f32x2(v[lg][2 * e], v[lg][2 * e + 1]);
              const uint64_t y =
                  a.residual ? fma_f32x2(a2f[lg][e & 1], acc2x,
                                         f32x2(pk[e] << 16, pk[e] & 0xFFFF0000u))
                             : mul_f32x2(a2f[lg][e & 1], acc2x);
              pk[e] = pack_bf16x2(__uint_as_float(static_cast<uint32_t>(y)),
                                  __uint_as_float(static_cast<uint32_t>(y >> 32)));
            }
            if (a.relu) {
#pragma unroll
              for (int e = 0; e < 8; ++e) pk[e] = relu_bf16x2(pk[e]);
            }
#pragma unroll
            for (int bp = 0; bp < 2; ++bp)
              stmatrix_x4_trans(addr[bp], pk[4 * bp + 0], pk[4 * bp + 1], pk[4 * bp + 2],
                                pk[4 * bp + 3]);
          }
        }
        if (c_begin >= c_end) {
          tc_fence_before_sync();
          mbar_arrive(&ctl->acc_empty[ab]);
        }
      } else if constexpr (kPoolBW == 0) {
        const int T = a.bw * a.bh * a.bn;
        const int nchunks = (a.tile_n + 31) / 32;
        const int c_begin = (nchunks * half + kParts - 1) / kParts;
        const int c_end = (nchunks * (half + 1) + kParts - 1) / kParts;
        // direct-store path: pixel of chunk c_begin walked in column order
        int px0 = 32 * c_begin;
        int wi = px0 % a.bw, hi = (px0 / a.bw) % a.bh, ni = px0 / (a.bw * a.bh);
        for (int j = c_begin; j < c_end; ++j) {
          uint32_t v[32];
          tmem_ld_32x32b_x32(acc + static_cast<uint32_t>(32 * j), v);
          tmem_wait_ld();
          if (j == c_end - 1) {
            // this warp has read its part of the accumulator
            tc_fence_before_sync();
            mbar_arrive(&ctl->acc_empty[ab]);
          }
          if (a.partial != nullptr) {
            // split K (1x1 image): pixel px is image n0 + px; the raw sum of
            // this K range goes to partial[split][n][k]
            float* dst = a.partial + (static_cast<size_t>(tc.split) * a.N + tc.n0 + 32 * j) * a.K + k;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (kvalid && 32 * j + i < T && tc.n0 + 32 * j + i < a.N)
                dst[static_cast<size_t>(i) * a.K] = __uint_as_float(v[i]);
          } else if (a.bh * a.bn == 1 && a.P * a.N == 1) {
            // a run of pixels: outputs K apart from the tile's first pixel on
            const int left = min(T, a.Q - tc.q0) - 32 * j;   // pixels of this chunk and after
            const size_t o0 = static_cast<size_t>(tc.q0 + 32 * j) * a.K + k;
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += 8) {
              float res[8];
#pragma unroll
              for (int i = 0; i < 8; ++i)
                res[i] = a.residual && kvalid && i0 + i < left
                             ? load_residual(a, o0 + static_cast<size_t>(i0 + i) * a.K) : 0.0f;
#pragma unroll
              for (int i = 0; i < 8; ++i)
                if (kvalid && i0 + i < left)
                  store_out(a, o0 + static_cast<size_t>(i0 + i) * a.K,
                            a2 * __uint_as_float(v[i0 + i]), res[i]);
            }
          } else if (!a.residual) {
            // store by store: the batches below keep 24 more values, which spill
            // where producers take the registers (gathering modes: 65 -> 33
            // channels, 1x1, 14 x 14, batch 32, 21.3 us so, 15.4 here)
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const int q = tc.q0 + wi, p = tc.p0 + hi, n = tc.n0 + ni;
              if (kvalid && 32 * j + i < T && q < a.Q && p < a.P && n < a.N)
                store_out(a, ((static_cast<size_t>(n) * a.P + p) * a.Q + q) * a.K + k,
                          a2 * __uint_as_float(v[i]));
              if (++wi == a.bw) {
                wi = 0;
                if (++hi == a.bh) { hi = 0; ++ni; }
              }
            }
          } else {
            // eight pixels at a time: their residuals are all requested before
            // the first output is stored (a load behind each store, which may
            // alias it, cost a memory latency per pixel)
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += 8) {
              size_t o[8];
              bool in[8];
              float res[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const int q = tc.q0 + wi, p = tc.p0 + hi, n = tc.n0 + ni;
                in[i] = kvalid && 32 * j + i0 + i < T && q < a.Q && p < a.P && n < a.N;
                o[i] = ((static_cast<size_t>(n) * a.P + p) * a.Q + q) * a.K + k;
                if (++wi == a.bw) {
                  wi = 0;
                  if (++hi == a.bh) { hi = 0; ++ni; }
                }
              }
#pragma unroll
              for (int i = 0; i < 8; ++i)
                res[i] = in[i] && a.residual ? load_residual(a, o[i]) : 0.0f;
#pragma unroll
              for (int i = 0; i < 8; ++i)
                if (in[i]) store_out(a, o[i], a2 * __uint_as_float(v[i0 + i]), res[i]);
            }
          }
        }
        if (c_begin >= c_end) {
          tc_fence_before_sync();
          mbar_arrive(&ctl->acc_empty[ab]);
        }
      } else if constexpr (kPoolBW == 1) {
        // fused 2x2 max pool of rows of any width a.bw: items of eight pooled
        // outputs of one row pair, 16 columns of each row per load (columns
        // past the row are read and not used; all 512 are allocated)
        const int Qp = a.bw / 2, groups = (Qp + 7) / 8, bh2 = a.bh / 2;
        const int items = a.bh * a.bn / 2 * groups;
        for (int it = half; it < items; it += 2) {
          const int pair = it / groups, g = it - pair * groups;
          uint32_t v0[16], v1[16];
          const uint32_t col = acc + static_cast<uint32_t>(pair * 2 * a.bw + 16 * g);
          tmem_ld_32x32b_x16(col, v0);
          tmem_ld_32x32b_x16(col + static_cast<uint32_t>(a.bw), v1);
          tmem_wait_ld();
          const int ni = pair / bh2, p2 = tc.p0 / 2 + pair - ni * bh2, n = tc.n0 + ni;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int q2 = 8 * g + j;
            // alpha >= 0, so max commutes with the scaling (and with ReLU)
            float mx = a2 * fmaxf(fmaxf(__uint_as_float(v0[2 * j]), __uint_as_float(v0[2 * j + 1])),
                                  fmaxf(__uint_as_float(v1[2 * j]), __uint_as_float(v1[2 * j + 1])));
            if (q2 >= Qp) continue;
            if (kTmaStore) {
              if (a.relu) mx = fmaxf(mx, 0.0f);
              stage[(pair * Qp + q2) * kBM + m] = __float2bfloat16_rn(mx);
            } else if (kvalid && p2 < Po && q2 < Qo && n < a.N) {
              store_out(a, ((static_cast<size_t>(n) * Po + p2) * Qo + q2) * a.K + k, mx);
            }
          }
        }
        tc_fence_before_sync();
        mbar_arrive(&ctl->acc_empty[ab]);
      } else {
        // fused 2x2 max pool: tiles hold whole rows of width kPoolBW (q0 = 0)
        // and an even number of rows per image; one TMEM load covers an even
        // pair of rows or more.
        constexpr int kCols = kPoolBW <= 16 ? 32 : 64;   // columns per load
        constexpr int kPairs = kCols / (2 * kPoolBW);    // row pairs per load
        const int rows_total = a.bh * a.bn;               // tile rows (all images)
        const int bh2 = a.bh / 2;
        const int nloads = (rows_total * kPoolBW + kCols - 1) / kCols;
        const int l_begin = half ? (nloads + 1) / 2 : 0;
        const int l_end = half ? nloads : (nloads + 1) / 2;
        for (int j = l_begin; j < l_end; ++j) {
          uint32_t v[kCols];
          tmem_ld_32x32b_x32(acc + static_cast<uint32_t>(kCols * j),
                             *reinterpret_cast<uint32_t(*)[32]>(v));
          if constexpr (kCols == 64)
            tmem_ld_32x32b_x32(acc + static_cast<uint32_t>(kCols * j + 32),
                               *reinterpret_cast<uint32_t(*)[32]>(v + 32));
          tmem_wait_ld();
          if (j == l_end - 1) {
            tc_fence_before_sync();
            mbar_arrive(&ctl->acc_empty[ab]);
          }
#pragma unroll
          for (int pp = 0; pp < kPairs; ++pp) {
            const int pair = j * kPairs + pp;          // row pair within the tile
            const int ni = pair / bh2;
            const int hi2 = pair - ni * bh2;
            const int p2 = tc.p0 / 2 + hi2, n = tc.n0 + ni;
            const bool pv = ni < a.bn;
#pragma unroll
            for (int q2 = 0; q2 < kPoolBW / 2; ++q2) {
              const int c0 = pp * 2 * kPoolBW + 2 * q2;
              const float m0 = fmaxf(__uint_as_float(v[c0]), __uint_as_float(v[c0 + 1]));
              const float m1 = fmaxf(__uint_as_float(v[c0 + kPoolBW]),
                                     __uint_as_float(v[c0 + kPoolBW + 1]));
              // alpha >= 0, so max commutes with the scaling (and with ReLU)
              float mx = a2 * fmaxf(m0, m1);
              if (kTmaStore) {
                if (pv) {
                  if (a.relu) mx = fmaxf(mx, 0.0f);
                  stage[(pair * (kPoolBW / 2) + q2) * kBM + m] = __float2bfloat16_rn(mx);
                }
              } else if (kvalid && pv && p2 < Po && q2 < Qo && n < a.N) {
                store_out(a, ((static_cast<size_t>(n) * Po + p2) * Qo + q2) * a.K + k, mx);
              }
            }
          }
        }
        if (l_begin >= l_end) {
          tc_fence_before_sync();
          mbar_arrive(&ctl->acc_empty[ab]);
        }
      }
      if (kTmaStore) {
        fence_proxy_async_smem();   // staged values -> visible to the TMA store
        named_barrier_sync(1, 32 * epi_warps(kMode));
        if (elected && ok) {
          if (kPoolBW) {
            tma_store_4d(&tmap_y, stage, tc.ktile * kBM, 0, tc.p0 / 2, tc.n0);
          } else if constexpr (kRowPair) {
            tma_store_4d(&tmap_y, stage, 0, 0, 0, tc.p0);
            tma_store_4d(&tmap_y, reinterpret_cast<uint8_t*>(stage) + 32768, 0, 0, 1, tc.p0);
          } else {
            tma_store_4d(&tmap_y, stage, tc.ktile * kBM, tc.q0, tc.p0, tc.n0);
            if (tc.ktile * kBM + kBM / 2 < a.K)
              tma_store_4d(&tmap_y, reinterpret_cast<uint8_t*>(stage) + 32768,
                           tc.ktile * kBM + kBM / 2, tc.q0, tc.p0, tc.n0);
          }
          bulk_commit_group();
        }
      }
    }
    if (kTmaStore && elected) bulk_wait_group<0>();   // all stores complete before exit
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
  }
  if constexpr (kCanCluster) {
    if (a.cluster) {
      grid_dependency_wait();   // for every thread: the residual is read, y written
      add_cluster_sums(a);
    }
  }
}


// ---------------------------------------------------------------- host side

inline int ceil_div(int64_t a, int64_t b) { return static_cast<int>((a + b - 1) / b); }

// TMA activations: whole 64-channel boxes, or 32-channel boxes in pairs.
inline bool use_tma(const ConvProblem& p) { return p.C % (kBK / 2) == 0 && p.sh <= 2 && p.sw <= 2; }
inline bool use_ch32(const ConvProblem& p) { return p.C % kBK != 0; }
// Output pixels per tile: whole rows of the output (so one TMA box per tap
// covers the tile), balanced so the last tile along each axis is not a
// sliver, at most 256 pixels.  With a fused 2x2 pool a tile holds whole
// output rows and an even number of them per image.
inline TilePlan plan_tiles(const ConvProblem& p, bool tma) {
  TilePlan t{};
  const int stride_w = tma ? static_cast<int>(p.sw) : 1;
  const int stride_h = tma ? static_cast<int>(p.sh) : 1;
  const int bw_max = static_cast<int>(std::min<int64_t>(p.Q, kMaxTileN / stride_w));
  t.tiles_q = ceil_div(p.Q, bw_max);
  t.bw = ceil_div(p.Q, t.tiles_q);
  if (t.tiles_q > 1) {
    t.bh = 1;
    t.bn = 1;
  } else {
    int bh_max = static_cast<int>(std::min<int64_t>({p.P, kMaxTileN / t.bw, 256 / stride_h}));
    if (p.pool) bh_max &= ~1;
    if (bh_max < 1) bh_max = 1;
    const int tp = ceil_div(p.P, bh_max);
    t.bh = ceil_div(p.P, tp);
    if (p.pool && (t.bh & 1)) t.bh += 1;   // <= bh_max when bh_max is even
    if (t.bh < p.P) {
      t.bn = 1;
    } else {
      t.bh = static_cast<int>(p.P) + (p.pool ? static_cast<int>(p.P & 1) : 0);
      const int bn_max = std::max(1, static_cast<int>(std::min<int64_t>(p.N, kMaxTileN / (t.bw * t.bh))));
      t.bn = ceil_div(p.N, ceil_div(p.N, bn_max));
    }
  }
  t.tiles_p = ceil_div(p.P, t.bh);
  t.tiles_n = ceil_div(p.N, t.bn);
  t.T = t.bw * t.bh * t.bn;
  t.tile_n = ((t.T + 15) / 16) * 16;
  t.im2col = t.rowpair = false;
  t.oN = p.N;
  t.oP = p.P;
  t.oQ = p.Q;
  return t;
}

// Patch mode (gathered activations staged per tile in shared memory) when a
// tile is whole output rows of one image, the filter spans at most
// kPatchMaxKBlocks K blocks and two patches fit beside the ring: the bytes of
// a patch buffer, else 0.
inline int patch_bytes_of(const ConvProblem& p, const TilePlan& t) {
  if (t.tiles_q != 1 || t.bn != 1) return 0;
  const int64_t kblocks = (p.C * p.R * p.S + kBK - 1) / kBK;
  if (kblocks > kPatchMaxKBlocks) return 0;
  const int64_t rows = static_cast<int64_t>(t.bh - 1) * p.sh + p.R;
  const int64_t elems = rows * (p.W + 2 * p.pw) * p.C;
  const int64_t cap = ((2 * elems + 32) + 15) / 16 * 16;
  if (cap > (int64_t(1) << 20)) return 0;
  if (smem_bytes_for(kModePatch, static_cast<size_t>(cap), static_cast<int>(kblocks)) >
      static_cast<size_t>(kSmemLimit))
    return 0;
  return static_cast<int>(cap);
}

// Whether padded boxes beat the modes whose threads build the operand.  They do
// at every channel count but 8 and 24: a tap's box is a K block of its own
// there, where 64 codes hold eight or nearly three taps, and rows of 16 or 48
// bytes are copied slowly (2.6 and 3.3 ns a pixel).  For those two the
// estimates decide, in ns and fitted to 58 layers: a gathered K block 1250 (700
// up to 128 pixels), a patch 4750 a tile and stride and 600 + 120 C a K block
// of 256 pixels.  (Batch 64, 32 x 32, 64 filters, padded and else: 8 channels 3
// x 3 16.4 and 16.4 us, 5 x 5 37.1 and 21.9; 24 channels 5 x 5 32 and 45, 7 x 7
// 60 and 48.)
inline bool pad_boxes_pay(const ConvProblem& p) {
  if ((p.C != 8 && p.C != 24) || p.R * p.S == 1) return true;
  const TilePlan t = plan_tiles(p, false);
  // only these widths pool without boxes
  if (p.pool && (t.tiles_q != 1 || t.T > kMaxTileN || (t.bh & 1) ||
                 (t.bw != 8 && t.bw != 16 && t.bw != 32)))
    return true;
  const int64_t sms = device_sm_count(), tk = ceil_div(p.K, kBM), px = p.N * p.P * p.Q;
  const int64_t kb = (p.C * p.R * p.S + kBK - 1) / kBK;
  const int64_t tiles = static_cast<int64_t>(t.tiles_q) * t.tiles_p * t.tiles_n * tk;
  const double built =
      patch_bytes_of(p, t) > 0
          ? 4750.0 * static_cast<double>(p.sh) +
                static_cast<double>(kb) * (600.0 + 120.0 * static_cast<double>(p.C)) * t.tile_n / kMaxTileN
          : 1500.0 + static_cast<double>(kb) * (t.tile_n > 128 ? 1250.0 : 700.0);
  const int64_t T = std::min<int64_t>(kMaxTileN, std::max<int64_t>(16, ((px * tk + sms - 1) / sms + 15) / 16 * 16));
  const double row = (p.C == 8 ? 2.6 : 3.3) * (p.sh == 1 ? 1.0 : 0.86);
  const double boxes = static_cast<double>(p.R * p.S) * std::max(250.0, row * static_cast<double>(T)) + 1500.0;
  return static_cast<double>(((px + T - 1) / T * tk + sms - 1) / sms) * boxes <=
         static_cast<double>((tiles + sms - 1) / sms) * built;
}

// Other multiples of 8 channels: 64-channel boxes, each tap's last one padded.
inline bool use_tma_pad(const ConvProblem& p) {
  return !use_tma(p) && p.C % 8 == 0 && p.sh <= 2 && p.sw <= 2 && p.ph <= p.R && p.pw <= p.S &&
         pad_boxes_pay(p);
}
inline bool tma_fed(const ConvProblem& p) { return use_tma(p) || use_tma_pad(p); }
inline int64_t kblocks_of(const ConvProblem& p) {
  return use_tma_pad(p) ? p.R * p.S * ((p.C + kBK - 1) / kBK)
                        : (p.C * p.R * p.S + kBK - 1) / kBK;
}

inline TilePlan plan_tiles(const ConvProblem& p) { return plan_tiles(p, tma_fed(p)); }

// The kernel's kPoolBW for a plan: -1 where a tile cannot pool (whole rows,
// an even number of them); 1 for rows of other widths than 8, 16 and 32,
// which the TMA-fed modes alone take (the explicit algorithm refuses them:
// conv_igemm_unsupported_reason).
inline int pool_width(const ConvProblem& p, const TilePlan& t) {
  if (!p.pool) return 0;
  if (t.tiles_q != 1 || t.T > kMaxTileN || (t.bh & 1)) return -1;
  if (t.bw == 8 || t.bw == 16 || t.bw == 32) return t.bw;
  return tma_fed(p) ? 1 : -1;
}

// Estimated time (ns) of a TMA-mode plan.  A K block of a T-pixel tile takes
// about 215 + 0.25 T ns on a CTA (fitted to the AlexNet and ResNet-18 layers:
// 256 ns at 176 pixels, 264 at 224, 285 at 256: supplying the operands costs
// nearly the same whatever the width), a tile about 0.9 us more, with a
// single accumulator, which its epilogue holds, 1.7 us.  CTAs take whole
// tiles, so what counts is the largest number any of them gets.
inline double plan_cost(const ConvProblem& p, const TilePlan& t, bool resident, int sms) {
  const int64_t tiles = static_cast<int64_t>(t.tiles_q) * t.tiles_p * t.tiles_n *
                        ((p.K + kBM - 1) / kBM);
  const double waves = static_cast<double>((tiles + sms - 1) / sms);
  const double kb = t.rowpair ? static_cast<double>((p.R + 1) * p.S * p.C / kBK)
                              : static_cast<double>(kblocks_of(p));
  const bool acc2 = !resident && t.tile_n <= kAcc2Cols;
  return waves * (kb * (215.0 + 0.25 * t.tile_n) + (acc2 ? 900.0 : 1700.0));
}

// Whether the activations can be fetched in im2col mode: the limits of the
// tensor map (corner offsets of a 4-D map are 8 bits, tap offsets unsigned),
// 32-bit pixel indices, and at least 128 KiB of input (smaller tensors are
// left to tiled boxes, which is where the one-image layers are).
inline bool im2col_ok(const ConvProblem& p) {
  return tma_fed(p) && p.R <= 128 && p.S <= 128 && p.ph <= 127 && p.pw <= 127 &&
         p.N * p.P * p.Q <= (int64_t(1) << 30) && p.N * p.H * p.W * p.C * 2 >= 131072 &&
         get_encode_im2col() != nullptr;
}

inline bool use_tma_store(const ConvProblem& p) {
  return p.ydt == TBN_BF16 && p.K % 8 == 0 && is_aligned(p.y, 16) &&
         (!p.residual || is_aligned(p.residual, 16));
}

// Whether the layer can run on row pairs (kModeRowPair): at most 64 filters,
// stride 1 down the rows, an even number of output rows of at most a tile's
// width, whole 64-channel boxes, and the staged bf16 epilogue.  It pays for
// filters of several rows: 3 x 3 over 64 channels takes 12 K blocks for two
// output rows instead of 18 (56 x 56 with shortcut, 64 filters, batch 64: 27.5
// us one row at a time, 22.2 in pairs; 24.6 when zero weights stood for the
// tap row that a half does not have and the epilogue looked for sums that an
// infinite input times those made NaN); plan_cost decides by the K blocks.
inline bool rowpair_ok(const ConvProblem& p) {
  return p.C % kBK == 0 && p.K <= kBM / 2 && p.sh == 1 && p.sw <= 2 && p.P % 2 == 0 && p.R >= 2 &&
         p.R < 128 && p.Q <= kMaxTileN && !p.pool && p.wq == nullptr && use_tma_store(p);
}

// The tile plan of a launch.  Gathering modes and split K: plan_tiles.  TMA
// modes: the cheapest (plan_cost) of plan_tiles, of runs of T consecutive
// pixels of the whole batch where im2col mode can fetch them (T a multiple
// of 16, or of two output rows when pooling), and otherwise of fewer rows per
// tile.  Whole-image tiles leave the last wave nearly empty (13 x 13 images,
// 384 filters, batch 256: 768 tiles on 152 SMs, six waves for 5.05) or their
// columns short of 256; runs of pixels are cut to the machine instead:
// four waves of 224 (that layer at 2304 codes per filter: 63.9 -> 50.6 us,
// at 3456: 91.4 -> 69.7; the AlexNet step at batch 256: 680 -> 627 us).
// `resident`: columns of tensor memory that each K block takes in the
// space-to-depth mode, where they all stay beside the accumulator (else 0).
// 24 instead of 32 columns for 48 channels leave room for tiles of 256 pixels
// instead of 224 (AlexNet conv1, batch 256: 79.4 -> 76.8 us; two accumulators
// beside them, of 144 pixels each, take 82 even with eight ring stages).
inline TilePlan plan_conv(const ConvProblem& p, int resident) {
  TilePlan best = plan_tiles(p);
  if (!tma_fed(p) || p.ksplit > 1) return best;
  const int sms = device_sm_count();
  double cost = plan_cost(p, best, resident, sms);
  const auto consider = [&](const TilePlan& t) {
    const double c = plan_cost(p, t, resident, sms);
    if (c < cost) {
      cost = c;
      best = t;
    }
  };
  const int kb = ceil_div(p.C * p.R * p.S, kBK);
  const int t_max = resident ? std::min(kMaxTileN, kTmemCols - resident * kb) : kMaxTileN;
  if (im2col_ok(p)) {
    TilePlan t = best;
    t.im2col = true;
    t.oN = 1;
    t.tiles_n = t.bn = 1;
    if (!p.pool) {
      t.oP = 1;
      t.oQ = p.N * p.P * p.Q;
      t.tiles_p = t.bh = 1;
      for (int T = 16; T <= t_max; T += 16) {
        t.T = t.bw = t.tile_n = T;
        t.tiles_q = ceil_div(t.oQ, T);
        consider(t);
      }
      if (rowpair_ok(p) && !resident) {
        // runs of whole row pairs
        t.rowpair = true;
        t.oP = p.N * p.P / 2;
        t.oQ = p.Q;
        t.bw = static_cast<int>(p.Q);
        t.tiles_q = 1;
        for (int rows = 1; rows * t.bw <= kMaxTileN; ++rows) {
          t.bh = rows;
          t.T = rows * t.bw;
          t.tile_n = ((t.T + 15) / 16) * 16;
          t.tiles_p = ceil_div(t.oP, rows);
          consider(t);
        }
      }
    } else if (p.P % 2 == 0 && best.tiles_q == 1) {
      // row pairs of all images in sequence (P even: none crosses images)
      t.oP = p.N * p.P;
      t.oQ = p.Q;
      t.bw = static_cast<int>(p.Q);
      t.tiles_q = 1;
      for (int rows = 2; rows * t.bw <= t_max; rows += 2) {
        t.bh = rows;
        t.T = rows * t.bw;
        t.tile_n = ((t.T + 15) / 16) * 16;
        t.tiles_p = ceil_div(t.oP, rows);
        consider(t);
      }
    }
  } else if (!p.pool && best.tiles_q == 1 && best.bn == 1) {
    TilePlan t = best;
    for (int rows = 1; rows < best.bh; ++rows) {
      t.bh = rows;
      t.T = t.bw * rows;
      t.tile_n = ((t.T + 15) / 16) * 16;
      t.tiles_p = ceil_div(p.P, rows);
      consider(t);
    }
  }
  return best;
}

// Output map: box = 128 filters x the tile's pixels (no swizzle), or with
// `halves`, 64 filters (128 bytes) per box with the 128-byte swizzle (the
// staging layout of the fragment epilogue, two stores per tile).
inline CUresult encode_out_map(CUtensorMap* m, const void* base, const ConvProblem& p, const TilePlan& t,
                        int pool, bool halves = false) {
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  if (t.rowpair) {
    // (filter, column, row parity, row pair)
    const cuuint64_t gd[4] = {(cuuint64_t)p.K, (cuuint64_t)t.oQ, 2u, (cuuint64_t)t.oP};
    const cuuint64_t gs[3] = {(cuuint64_t)(p.K * 2), (cuuint64_t)(t.oQ * p.K * 2),
                              (cuuint64_t)(2 * t.oQ * p.K * 2)};
    const cuuint32_t bx[4] = {(cuuint32_t)(kBM / 2), (cuuint32_t)t.bw, 1u, (cuuint32_t)t.bh};
    return get_encode_tiled()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gd,
                              gs, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  const int64_t Po = pool ? t.oP / 2 : t.oP, Qo = pool ? t.oQ / 2 : t.oQ;
  const cuuint64_t gdim[4] = {(cuuint64_t)p.K, (cuuint64_t)Qo, (cuuint64_t)Po, (cuuint64_t)t.oN};
  const cuuint64_t gstride[3] = {(cuuint64_t)(p.K * 2), (cuuint64_t)(Qo * p.K * 2),
                                 (cuuint64_t)(Po * Qo * p.K * 2)};
  const cuuint32_t box[4] = {(cuuint32_t)(halves ? kBM / 2 : kBM), (cuuint32_t)(pool ? t.bw / 2 : t.bw),
                             (cuuint32_t)(pool ? t.bh / 2 : t.bh), (cuuint32_t)t.bn};
  return get_encode_tiled()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gdim,
                            gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            halves ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int kMode, int kPoolBW, bool kTmaStore, bool kFuse>
tbn_status launch_t(const ConvProblem& p, const TilePlan& t, IgArgs& a, cudaStream_t s) {
  constexpr bool kGather = mode_gathers(kMode);
  constexpr bool kCh32 = kMode == kModeTma32;
  alignas(64) CUtensorMap tmap_x, tmap_y, tmap_res, tmap_x32;
  std::memset(&tmap_x, 0, sizeof(tmap_x));
  std::memset(&tmap_y, 0, sizeof(tmap_y));
  std::memset(&tmap_res, 0, sizeof(tmap_res));
  std::memset(&tmap_x32, 0, sizeof(tmap_x32));
  if (!kGather) {
    const cuuint64_t gdim[4] = {(cuuint64_t)p.C, (cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.N};
    const cuuint64_t gstride[3] = {(cuuint64_t)(p.C * 2), (cuuint64_t)(p.W * p.C * 2),
                                   (cuuint64_t)(p.H * p.W * p.C * 2)};
    // row pairs: base rows two apart, R + 1 tap rows
    const int rp = t.rowpair ? 1 : 0;
    const cuuint32_t estr[4] = {1u, (cuuint32_t)p.sw, (cuuint32_t)(p.sh + rp), 1u};
    // Boxes narrower than a pixel's channels, or than the 64 of a box, read
    // rows that do not fill 256-byte lines: promoting their requests to whole
    // ones reads beside what is wanted (27 x 27, batch 256, 96 -> 256 channels,
    // 5 x 5: 142 us so, 138 without; 40 -> 128 channels, batch 32, fp32 y: 26.3
    // and 22.2; layers of 64-channel boxes are within 1% either way).
    const CUtensorMapL2promotion promotion = kCh32 || kMode == kModeTapPair || kMode == kModeTmaPad
                                                 ? CU_TENSOR_MAP_L2_PROMOTION_NONE
                                                 : CU_TENSOR_MAP_L2_PROMOTION_L2_256B;
    const cuuint32_t box[4] = {0u, (cuuint32_t)(t.bw * p.sw), (cuuint32_t)(t.bh * p.sh),
                               (cuuint32_t)t.bn};
    if (!t.im2col && (box[1] > 256 || box[2] > 256 || box[3] > 256))
      return fail(TBN_ERR_UNSUPPORTED, "implicit GEMM: TMA box too large");
    const auto encode = [&](CUtensorMap* m, cuuint32_t channels) {
      const CUtensorMapSwizzle swizzle =
          channels == kBK ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
      if (t.im2col) {
        // base positions [-pad, size - 1 + pad - (kernel - 1)] in steps of the stride
        const int lower[2] = {-(int)p.pw, -(int)p.ph};
        const int upper[2] = {(int)(p.pw - (p.S - 1)), (int)(p.ph - (p.R - 1)) - rp};
        return get_encode_im2col()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                                   const_cast<void*>(p.x), gdim, gstride, lower, upper, channels,
                                   (cuuint32_t)t.T, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                                   promotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      }
      const cuuint32_t b[4] = {channels, box[1], box[2], box[3]};
      return get_encode_tiled()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p.x),
                                gdim, gstride, b, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                                promotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult cr = encode(&tmap_x, kCh32 ? kBK / 2 : kBK);
    if (cr == CUDA_SUCCESS && kMode == kModeTapPair) cr = encode(&tmap_x32, kBK / 2);
    if (cr != CUDA_SUCCESS) return fail(TBN_ERR_CUDA, "tensor map of x failed (%d)", (int)cr);
  }
  if (kTmaStore) {
    // the fragment epilogue (no pool) stages two swizzled halves
    const bool halves = kPoolBW == 0;
    CUresult cr = encode_out_map(&tmap_y, p.y, p, t, kPoolBW ? 1 : 0, halves);
    if (cr != CUDA_SUCCESS) return fail(TBN_ERR_CUDA, "cuTensorMapEncodeTiled(y) failed (%d)", (int)cr);
    if (p.residual) {
      cr = encode_out_map(&tmap_res, p.residual, p, t, 0, true);
      if (cr != CUDA_SUCCESS)
        return fail(TBN_ERR_CUDA, "cuTensorMapEncodeTiled(residual) failed (%d)", (int)cr);
    }
  }
  auto kern = conv_igemm_kernel<kMode, kPoolBW, kTmaStore, kFuse>;
  const size_t smem = smem_bytes_for(kMode, static_cast<size_t>(a.patch_cap), a.kblocks);
  // kernel attributes: set once per process (one process drives one GPU);
  // the shared-memory limit is the largest any launch of the mode can need
  static std::once_flag once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(once, [&] {
    attr_err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kSmemLimit);
    if (attr_err == cudaSuccess)
      attr_err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
  if (attr_err != cudaSuccess) return cuda_fail(attr_err, "cudaFuncSetAttribute(conv_igemm_kernel)");
  // fused quantization: one CTA per SM whatever the tile count, so that the
  // whole GPU quantizes (CTAs without a tile stop after the barrier)
  const int grid = kFuse ? device_sm_count() : std::min(a.tiles, device_sm_count());
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(threads_for<kMode>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  if (kFuse) {
    // fused quantization: the CTAs meet at a grid-wide barrier, so they must
    // all be resident at once
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  } else {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.cluster) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(a.ksplit);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    cfg.gridDim = dim3(static_cast<unsigned>(a.tiles));   // whole clusters, a tile each
  }
  if (kFuse) {
    const cudaError_t me = cudaMemsetAsync(a.gbar, 0, sizeof(unsigned), s);
    if (me != cudaSuccess) return cuda_fail(me, "cudaMemsetAsync(barrier word)");
  }
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kern, tmap_x, tmap_y, tmap_res, tmap_x32, a);
  if (le != cudaSuccess) return cuda_fail(le, "cudaLaunchKernelEx(conv_igemm_kernel)");
  return check_launch("conv_igemm_kernel");
}

template <int kMode, bool kTmaStore, bool kFuse>
tbn_status launch_pool(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw, cudaStream_t s) {
  switch (pw) {
    case 8: return launch_t<kMode, 8, kTmaStore, kFuse>(p, t, a, s);
    case 16: return launch_t<kMode, 16, kTmaStore, kFuse>(p, t, a, s);
    case 32: return launch_t<kMode, 32, kTmaStore, kFuse>(p, t, a, s);
    case 1:
      if constexpr (!mode_gathers(kMode) && !kFuse)
        return launch_t<kMode, 1, kTmaStore, kFuse>(p, t, a, s);
      return fail(TBN_ERR_UNSUPPORTED, "implicit GEMM: no pooled rows of this width");
    default: return launch_t<kMode, 0, kTmaStore, kFuse>(p, t, a, s);
  }
}

}  // namespace

// The per-mode launchers: pw = the fused pool's tile width (0: none),
// tma_store = the TMA-store epilogue, fuse = quantize the fp32 filters
// a.wq in the same (cooperative) launch.
tbn_status launch_igemm_tma64(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                              bool tma_store, bool fuse, cudaStream_t s);
// Clusters of `size` (2 .. kMaxCluster) CTAs of the TMA modes that the device
// runs at once (0: none).
int igemm_max_clusters(int size);
tbn_status launch_igemm_tma32(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                              bool tma_store, bool fuse, cudaStream_t s);
tbn_status launch_igemm_pad(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                            bool tma_store, cudaStream_t s);
tbn_status launch_igemm_tappair(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                                bool tma_store, bool fuse, cudaStream_t s);
tbn_status launch_igemm_rowpair(const ConvProblem& p, const TilePlan& t, IgArgs& a,
                                cudaStream_t s);

}  // namespace tbn
