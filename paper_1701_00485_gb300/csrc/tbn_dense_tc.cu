// tbn_dense_tc.cu -- the full-precision first convolution (fp32 weights, bf16
// NCHW input, bf16 NHWC output, even column stride: ResNet-18's 7x7/2 over 3
// channels) on the tensor cores, without giving up fp32 weights or sums.
//
// Arithmetic.  A fp32 weight is exactly the sum of three bf16 numbers (8 + 8 +
// 8 significand bits, cut off the top one after another), and a product of
// two bf16 numbers is exact in fp32.  So y = sum x h + sum x m + sum x l, three
// sums of exact products accumulated in fp32 by the tensor core and added in
// fp32: no weight bit is dropped (below bf16's smallest subnormal, 2^-133,
// aside), and the rounding error is that of fp32 sums, fewer of them than
// one per tap.  Where the result is not finite (an infinite or NaN input or
// weight, or an overflow) it is recomputed tap by tap in fp32, as the
// CUDA-core kernel does, because the split's zero terms times infinity are NaN.
// What that costs (32 images of 3 x 224 x 224, 37 us when finite, some 220 on
// the CUDA cores): 195 us for a batch of NaN, 297 of infinities, 2.6 ms where
// every sum overflows or most hold an infinity.
//
// GEMM view of a tile: D[128 pixels x 192] = A[128 x k] B[k x 192], where the
// 192 columns are 64 filters x {h, m, l} (one read of A serves all three) and
// k counts codes of 8 per (channel, filter row): the up to 8 taps of one
// filter row are 8 consecutive elements of one input row, starting at an even
// column (the column stride is even, so every pixel's run starts at the same
// parity; for odd padding one zero-weight tap in front makes it even), i.e.
// four aligned 32-bit words.
//   A   built by threads: one pixel (= tensor-memory lane) per thread reads
//       its four words per (channel, row) from the tile's input patch in
//       shared memory (consecutive lanes, consecutive words) and writes them
//       straight into a four-slot tensor-memory ring of 64 codes each.
//   B   the split weights, in shared memory for the whole launch (K-major,
//       128-byte swizzle).
//   D   two fp32 accumulators of 192 columns, so a tile's MMAs overlap the
//       previous tile's epilogue; epilogue threads (lane = pixel) add the
//       three terms, apply ReLU, and stage bf16 rows for one TMA store.
// A tile is 128 consecutive pixels of an image's output map; its input rows
// arrive by one TMA box, zero-filled outside the image.
//
// Bound and measured (7x7/2 over 3 x 224 x 224, batch 128): 83 us, where the
// CUDA-core kernel takes 871.  The MMAs need 96 cycles per 16 codes, 1056 per
// tile (46 us; shared memory is read for 528 + 336 of those cycles, the output
// write is 30 us of memory time), a tile takes about 1650.  What is left is
// the roles' serial instruction paths: with some 20 warps on an SM a warp
// issues about one instruction in ten cycles, so a hundred of them per block
// or tile is a thousand cycles.  That is why the coordinates are divided by
// multiplication, the chunk offsets come from a table, three groups of
// builders take turns (two: 103 us), the three terms are added two filters at
// a time, and the MMA warp issues a block as one predicated statement
// (before all that: 120 us).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "tbn_device.cuh"
#include "tbn_internal.h"

namespace tbn {
namespace {

constexpr int kPix = 128;                 // pixels per tile (MMA M)
constexpr int kFilt = 64;                 // filters per CTA
constexpr int kCols = 3 * kFilt;          // MMA N
constexpr int kSlots = 4;                 // A ring, 64 codes = 32 columns each
constexpr int kSlotCols = 32;
constexpr int kRingCol = 2 * kCols;       // accumulators [0, 192) and [192, 384)
constexpr int kTmemAll = 512;
constexpr int kPatches = 3;               // input patches in flight
constexpr int kBuildGroups = 3;           // groups of four warps (128 lanes) take blocks in turn
constexpr int kBuildWarps = 4 * kBuildGroups;
constexpr int kEpWarps = 8;               // two groups of four, 32 filters each
constexpr int kTmaWarp = kBuildWarps + kEpWarps;
constexpr int kMmaWarp = kTmaWarp + 1;
constexpr int kThreads = 32 * (kMmaWarp + 1);
constexpr int kWBlockBytes = kCols * 128; // 64 codes of the 192 columns
constexpr int kOutBytes = kPix * kFilt * 2;
constexpr int kMaxBlocks = 5;
constexpr int kSmemMax = 227 * 1024;
constexpr uint64_t kLimitNs = 1000000000ull;
static_assert(kRingCol + kSlots * kSlotCols <= kTmemAll, "tensor memory");

struct Args {
  FastDiv by_img, by_q;   // tiles_img, Q
  int C, H, W, K, R, S, sh, sw, ph, pw, Q, PQ;
  int tiles_img, tiles;   // tiles per image, in all
  int nch, blocks;        // (channel, row) chunks of 8 codes; 64-code blocks
  int lead;               // zero-weight taps in front of a row's S taps
  int prow_elems;         // patch row, elements
  int pplane_elems;       // patch plane (one channel), elements
  int patch_bytes;        // one patch (multiple of 128)
  int box_bytes;
  const __nv_bfloat16* x;
  const float* w;         // [K][C][R][S]
  int relu;
  uint32_t* err;
};

struct alignas(16) Ctl {
  // byte offsets in the patch of each (channel, row) chunk; those past the
  // last repeat it (their weights are zero)
  int chunk_off[8 * kMaxBlocks];
  uint64_t pfull[kPatches], pempty[kPatches];
  uint64_t full[kSlots], empty[kSlots];
  uint64_t dfull[2], dempty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

// Results that are not finite, tap by tap in fp32: bit i of `bad` is filter
// k + i of this lane's pixel `pix` of image n, staged in `row_s` (the pixel's
// 64 filters, 16-byte chunks permuted by `swz`) from chunk `chunk` on.  By the
// whole warp, eight filters at a time, so that a tap's weights are one load for
// all lanes and its input one load for eight filters; ends early when every
// sum that is needed is NaN.
__device__ __noinline__ void repair_by_taps(const Args& a, int n, int k, int pix, uint32_t bad,
                                            uint8_t* row_s, int chunk, int swz) {
  const int p = pix / a.Q, q = pix - p * a.Q;
  const int h0 = p * a.sh - a.ph, w0 = q * a.sw - a.pw, wstep = a.nch * a.S;
  for (int g = 0; g < 4; ++g, bad >>= 8, k += 8) {   // K % 8 == 0
    const bool need = (bad & 0xFFu) != 0u;
    if (!__any_sync(0xffffffffu, need)) continue;
    const float* wk = a.w + static_cast<int64_t>(k) * wstep;
    float acc[8] = {};
    for (int cr = 0; cr < a.nch; ++cr) {
      const int c = cr / a.R, h = h0 + cr - c * a.R;
      const __nv_bfloat16* xr = a.x + ((static_cast<int64_t>(n) * a.C + c) * a.H + h) * a.W + w0;
      const bool hv = h >= 0 && h < a.H;
#pragma unroll 4
      for (int s = 0; s < a.S; ++s) {
        const float xv = hv && w0 + s >= 0 && w0 + s < a.W ? __bfloat162float(xr[s]) : 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          acc[j] = fmaf(xv, __ldg(wk + j * wstep + cr * a.S + s), acc[j]);
      }
      bool done = true;
#pragma unroll
      for (int j = 0; j < 8; ++j) done &= acc[j] != acc[j];
      if (__all_sync(0xffffffffu, done || !need)) break;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if ((bad >> j) & 1u) {
        const float v = a.relu ? fmaxf(acc[j], 0.0f) : acc[j];   // NaN gives 0 there
        reinterpret_cast<__nv_bfloat16*>(row_s + (((chunk + g) ^ swz) << 4))[j] =
            __float2bfloat16_rn(v);
      }
  }
  __syncwarp();
}

__global__ void __launch_bounds__(kThreads, 1)
    dense_conv_tc_kernel(const __grid_constant__ CUtensorMap tmap_x,
                         const __grid_constant__ CUtensorMap tmap_y,
                         const __grid_constant__ Args a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* w_s = smem;                                        // [blocks][192 rows][128 B]
  uint8_t* out_s = w_s + a.blocks * kWBlockBytes;             // 2 x 16 KiB
  uint8_t* patch_s = out_s + 2 * kOutBytes;                   // kPatches patches
  Ctl* ctl = reinterpret_cast<Ctl*>(patch_s + kPatches * a.patch_bytes);
  volatile int* abort_flag = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = blockIdx.y * kFilt;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kPatches; ++i) {
      mbar_init(&ctl->pfull[i], 1);
      mbar_init(&ctl->pempty[i], 32 * kBuildWarps);
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&ctl->full[i], kPix);
      mbar_init(&ctl->empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&ctl->dfull[i], 1);
      mbar_init(&ctl->dempty[i], 32 * kEpWarps);
    }
    mbar_init(&ctl->drain, 1);
    ctl->abort = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_x);
    prefetch_tmap(&tmap_y);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&ctl->tmem_base, kTmemAll);
    tmem_relinquish();
  }
  for (int i = threadIdx.x; i < 8 * a.blocks; i += kThreads) {
    const int ch = min(i, a.nch - 1), c = ch / a.R;
    ctl->chunk_off[i] = 2 * (c * a.pplane_elems + (ch - c * a.R) * a.prow_elems);
  }
  // the weights' three terms: row f + 64 t of block b holds term t of filter
  // k0 + f, codes [64 b, + 64): chunk of 8 per (channel, row), tap s at
  // position lead + s, zero elsewhere
  for (int i = threadIdx.x; i < kFilt * a.blocks * 8; i += kThreads) {
    const int f = i % kFilt, ch = i / kFilt, k = k0 + f;
    const bool in = k < a.K && ch < a.nch;
    const float* wr = a.w + (static_cast<int64_t>(in ? k : 0) * a.nch + (in ? ch : 0)) * a.S;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int s = j - a.lead;
      v[j] = (in && s >= 0 && s < a.S) ? __ldg(wr + s) : 0.0f;
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      uint32_t pk[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t b0 = __float_as_uint(v[2 * j]) & 0xFFFF0000u;
        const uint32_t b1 = __float_as_uint(v[2 * j + 1]) & 0xFFFF0000u;
        v[2 * j] -= __uint_as_float(b0);       // exact
        v[2 * j + 1] -= __uint_as_float(b1);
        pk[j] = (b0 >> 16) | b1;
      }
      const int row = t * kFilt + f;
      *reinterpret_cast<uint4*>(w_s + (ch >> 3) * kWBlockBytes + row * 128 +
                                (((ch & 7) ^ (row & 7)) << 4)) =
          make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
  }
  fence_proxy_async_smem();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  // all 512 columns are allocated, so the base can only be 0; anything else
  // is reported and the CTA does no work
  if (ctl->tmem_base != 0u) {
    if (threadIdx.x == 0) raise_device_error(a.err, TBN_DEVERR_BAD_LAUNCH);
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(ctl->tmem_base, kTmemAll);
    return;
  }

  if (warp == kTmaWarp) {
    // ---------------- input patches
    int i = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++i) {
      const int b = i % kPatches;
      ok = mbar_wait(&ctl->pempty[b], (static_cast<uint32_t>(i / kPatches) & 1u) ^ 1u, abort_flag,
                     a.err, kLimitNs);
      if (!__all_sync(0xffffffffu, ok)) break;
      const int n = a.by_img(t), p0 = a.by_q((t - n * a.tiles_img) * kPix);
      if (elect_one()) {
        mbar_arrive_expect_tx(&ctl->pfull[b], static_cast<uint32_t>(a.box_bytes));
        tma_load_4d(patch_s + b * a.patch_bytes, &tmap_x, &ctl->pfull[b], -8,
                    p0 * a.sh - a.ph, 0, n);
      }
      __syncwarp();
    }
    // every copy issued must land before the CTA may exit
    for (int j = i > kPatches ? i - kPatches : 0; j < i; ++j)
      mbar_wait(&ctl->pfull[j % kPatches], static_cast<uint32_t>(j / kPatches) & 1u, nullptr,
                a.err, kLimitNs);
  } else if (warp == kMmaWarp) {
    // ---------------- MMA issue
    const uint32_t idesc = idesc_bf16_f32(kPix, kCols);
    const uint64_t wdesc = smem_desc_sw128_kmajor(smem_addr(w_s));
    int issued = 0;
    uint32_t i = 0, sl = 0, ph = 0;   // ring slot and the parity of its fill
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++i) {
      const uint32_t db = i & 1u;
      ok = mbar_wait_warp(&ctl->dempty[db], ((i >> 1) & 1u) ^ 1u, abort_flag, a.err, kLimitNs);
      if (!ok) break;
      for (int b = 0; b < a.blocks; ++b) {
        ok = mbar_wait_warp(&ctl->full[sl], ph, abort_flag, a.err, kLimitNs);
        if (!ok) break;
        tc_fence_after_sync();
        tc_mma_ts_block<2, 4, 6>(db * kCols, kRingCol + sl * kSlotCols,
                        wdesc + static_cast<uint64_t>(b * (kWBlockBytes >> 4)), idesc,
                        b != 0 ? 1u : 0u, (a.nch - 8 * b + 1) / 2, &ctl->empty[sl],
                        b == a.blocks - 1 ? &ctl->dfull[db] : nullptr);
        ++issued;
        if (++sl == kSlots) {
          sl = 0;
          ph ^= 1u;
        }
      }
    }
    if (!ok && issued > 0) {
      // in-flight MMAs end before tensor memory is freed
      if (elect_one()) tc_commit(&ctl->drain);
      __syncwarp();
      mbar_wait(&ctl->drain, 0u, nullptr, a.err, kLimitNs);
    }
  } else if (warp < kBuildWarps) {
    // ---------------- A rows: this thread's pixel, blocks g % kBuildGroups == group
    const int group = warp >> 2, px = (warp & 3) * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int row_b = a.prow_elems * 2;
    const int col0 = 2 * (8 - a.pw - a.lead);
    uint32_t g = static_cast<uint32_t>(group), pb = 0, pph = 0;
    int b = group;   // this group's next block within the tile
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
      ok = mbar_wait(&ctl->pfull[pb], pph, abort_flag, a.err, kLimitNs);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      const int f0 = (t - a.by_img(t) * a.tiles_img) * kPix;
      const int pix = min(f0 + px, a.PQ - 1);   // pixels past the map repeat its last one
      const int p = a.by_q(pix), q = pix - p * a.Q;
      const uint32_t base = smem_addr(patch_s + pb * a.patch_bytes) +
                            static_cast<uint32_t>((p - a.by_q(f0)) * a.sh * row_b +
                                                  2 * q * a.sw + col0);
      for (; b < a.blocks; b += kBuildGroups, g += kBuildGroups) {
        int off[8];
        *reinterpret_cast<int4*>(off) = *reinterpret_cast<const int4*>(&ctl->chunk_off[8 * b]);
        *reinterpret_cast<int4*>(off + 4) = *reinterpret_cast<const int4*>(&ctl->chunk_off[8 * b + 4]);
        uint32_t v[32];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v[4 * j + u]) : "r"(base + off[j] + 4 * u));
        const uint32_t sl = g % kSlots;
        ok = mbar_wait(&ctl->empty[sl], ((g / kSlots) & 1u) ^ 1u, abort_flag, a.err, kLimitNs);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        tc_fence_after_sync();
        tmem_st_32x32b_x32(lane_off + kRingCol + sl * kSlotCols, v);
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(&ctl->full[sl]);
      }
      b -= a.blocks;
      if (ok) mbar_arrive(&ctl->pempty[pb]);
      if (++pb == kPatches) {
        pb = 0;
        pph ^= 1u;
      }
    }
  } else {
    // ---------------- epilogue: this thread's pixel, filters [32 half, + 32)
    const int ew = warp - kBuildWarps, sub = ew & 3, half = ew >> 2;
    const int row = sub * 32 + lane;
    const bool elected = threadIdx.x == 32 * kBuildWarps;
    const uint32_t lane_off = static_cast<uint32_t>(sub * 32) << 16;
    uint32_t i = 0;
    bool ok = true;
    // the warps meet at named barriers: after a failed wait they keep
    // walking the tiles without working
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++i) {
      const uint32_t db = i & 1u;
      uint8_t* stage = out_s + db * kOutBytes;
      if (elected) bulk_wait_group_read<1>();   // the store of two tiles ago has been read
      named_barrier_sync(1, 32 * kEpWarps);
      if (ok) ok = mbar_wait(&ctl->dfull[db], (i >> 1) & 1u, abort_flag, a.err, kLimitNs);
      ok = __all_sync(0xffffffffu, ok);
      const int n = a.by_img(t), f0 = (t - n * a.tiles_img) * kPix;
      if (ok) {
        tc_fence_after_sync();
        uint32_t bad = 0;   // results that are not finite
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          uint32_t vh[16], vm[16], vl[16];
          const uint32_t col = lane_off + db * kCols + static_cast<uint32_t>(32 * half + 16 * cc);
          tmem_ld_32x32b_x16(col, vh);
          tmem_ld_32x32b_x16(col + kFilt, vm);
          tmem_ld_32x32b_x16(col + 2 * kFilt, vl);
          tmem_wait_ld();
          if (cc == 1) {
            tc_fence_before_sync();
            mbar_arrive(&ctl->dempty[db]);
          }
          // (l + m) + h; zero times the results sums to zero unless one of
          // them is infinite or NaN
          uint64_t o2[8], zero = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            o2[j] = add_f32x2(add_f32x2(f32x2(vl[2 * j], vl[2 * j + 1]),
                                        f32x2(vm[2 * j], vm[2 * j + 1])),
                              f32x2(vh[2 * j], vh[2 * j + 1]));
            zero = fma_f32x2(o2[j], 0ull, zero);
          }
          float o[16];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            o[2 * j] = __uint_as_float(static_cast<uint32_t>(o2[j]));
            o[2 * j + 1] = __uint_as_float(static_cast<uint32_t>(o2[j] >> 32));
          }
          const float z = __uint_as_float(static_cast<uint32_t>(zero)) +
                          __uint_as_float(static_cast<uint32_t>(zero >> 32));
          // one decision for the warp: collective instructions follow
          if (__any_sync(0xffffffffu, z != 0.0f)) {   // NaN != 0
#pragma unroll
            for (int j = 0; j < 16; ++j)
              bad |= (fabsf(o[j]) <= 3.402823466e38f ? 0u : 1u) << (16 * cc + j);
          }
          uint32_t pk[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            pk[j] = a.relu ? pack_bf16x2_relu(o[2 * j], o[2 * j + 1])
                           : pack_bf16x2(o[2 * j], o[2 * j + 1]);
#pragma unroll
          for (int u = 0; u < 2; ++u)
            *reinterpret_cast<uint4*>(stage + row * 128 +
                                      (((4 * half + 2 * cc + u) ^ (row & 7)) << 4)) =
                make_uint4(pk[4 * u], pk[4 * u + 1], pk[4 * u + 2], pk[4 * u + 3]);
        }
        const int k = k0 + 32 * half;
        bad = f0 + row < a.PQ && k < a.K ? bad & (0xFFFFFFFFu >> max(0, k + 32 - a.K)) : 0u;
        if (__any_sync(0xffffffffu, bad != 0u))
          repair_by_taps(a, n, k, min(f0 + row, a.PQ - 1), bad, stage + row * 128, 4 * half,
                         row & 7);
      }
      fence_proxy_async_smem();
      named_barrier_sync(1, 32 * kEpWarps);
      if (elected && ok) {
        tma_store_4d(&tmap_y, stage, k0, f0, n, 0);   // clipped at the map's end and at K
        bulk_commit_group();
      }
    }
    if (elected) bulk_wait_group<0>();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(0, kTmemAll);
  }
}

// The launch's shape, false where the kernel does not apply.
bool plan(const ConvProblem& p, Args* out, size_t* smem) {
  if (p.layout != TBN_NCHW_NHWC || p.xdt != TBN_BF16 || p.ydt != TBN_BF16) return false;
  // TMA: 16-byte rows of x, filters of y; aligned runs: an even column stride
  if (p.W % 8 != 0 || p.K % 8 != 0 || !is_aligned(p.x, 16) || !is_aligned(p.y, 16)) return false;
  if (p.sw % 2 != 0 || p.sw > 16 || p.sh > 64) return false;
  Args a{};
  a.lead = static_cast<int>(p.pw & 1);
  if (p.S + a.lead > 8 || p.pw + a.lead > 8) return false;
  if (p.C * p.R > 8 * kMaxBlocks || p.ph > 64) return false;
  if (p.P * p.Q > (int64_t(1) << 30) || p.H > (1 << 20) || p.W > (1 << 20) || p.K > (1 << 20)) return false;
  const int64_t pcols = ((p.Q - 1) * p.sw + 8 - p.pw - a.lead + 8 + 7) / 8 * 8;
  const int64_t prows = (p.Q - 1 + kPix - 1) / p.Q * p.sh + p.R;
  if (pcols > 256 || prows > 256) return false;
  a.C = (int)p.C; a.H = (int)p.H; a.W = (int)p.W; a.K = (int)p.K; a.R = (int)p.R; a.S = (int)p.S;
  a.sh = (int)p.sh; a.sw = (int)p.sw; a.ph = (int)p.ph; a.pw = (int)p.pw;
  a.Q = (int)p.Q; a.PQ = (int)(p.P * p.Q);
  a.tiles_img = (a.PQ + kPix - 1) / kPix;
  a.by_img = fast_div(a.tiles_img);
  a.by_q = fast_div(a.Q);
  if (p.N * a.tiles_img > 0x7fffffffLL) return false;
  a.tiles = (int)(p.N * a.tiles_img);
  a.nch = (int)(p.C * p.R);
  a.blocks = (a.nch + 7) / 8;
  a.prow_elems = (int)pcols;
  a.pplane_elems = (int)(pcols * prows);
  a.box_bytes = (int)(pcols * prows * p.C * 2);
  a.patch_bytes = (a.box_bytes + 127) / 128 * 128;
  *smem = 1024 + static_cast<size_t>(a.blocks) * kWBlockBytes + 2 * kOutBytes +
          static_cast<size_t>(kPatches) * a.patch_bytes + sizeof(Ctl);
  if (*smem > static_cast<size_t>(kSmemMax)) return false;
  *out = a;
  return true;
}

}  // namespace

// Taken wherever it applies: at batch 128 of the 7x7/2 layer over 3 x 224 x
// 224 it replaces the CUDA-core kernel's 870 us.
bool dense_conv_tc_takes(const ConvProblem& p) {
  Args a;
  size_t smem;
  return get_encode_tiled() != nullptr && plan(p, &a, &smem);
}

tbn_status launch_dense_conv_tc(const ConvProblem& p, const float* w, cudaStream_t s) {
  Args a;
  size_t smem = 0;
  if (!plan(p, &a, &smem)) return fail(TBN_ERR_UNSUPPORTED, "dense conv: not a tensor-core shape");
  a.x = static_cast<const __nv_bfloat16*>(p.x);
  a.w = w;
  a.relu = p.relu;
  a.err = device_error_word();
  alignas(64) CUtensorMap tmap_x, tmap_y;
  std::memset(&tmap_x, 0, sizeof(tmap_x));
  std::memset(&tmap_y, 0, sizeof(tmap_y));
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  {
    const cuuint64_t gdim[4] = {(cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.C, (cuuint64_t)p.N};
    const cuuint64_t gstr[3] = {(cuuint64_t)(p.W * 2), (cuuint64_t)(p.H * p.W * 2),
                                (cuuint64_t)(p.C * p.H * p.W * 2)};
    const cuuint32_t box[4] = {(cuuint32_t)a.prow_elems,
                               (cuuint32_t)(a.pplane_elems / a.prow_elems), (cuuint32_t)p.C, 1u};
    const CUresult cr = get_encode_tiled()(
        &tmap_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p.x), gdim, gstr, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) return fail(TBN_ERR_CUDA, "dense conv: tensor map of x failed (%d)", (int)cr);
  }
  {
    const cuuint64_t gdim[4] = {(cuuint64_t)p.K, (cuuint64_t)a.PQ, (cuuint64_t)p.N, 1u};
    const cuuint64_t gstr[3] = {(cuuint64_t)(p.K * 2), (cuuint64_t)(p.K * 2 * a.PQ),
                                (cuuint64_t)(p.K * 2 * a.PQ * p.N)};
    const cuuint32_t box[4] = {(cuuint32_t)kFilt, (cuuint32_t)kPix, 1u, 1u};
    const CUresult cr = get_encode_tiled()(
        &tmap_y, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, p.y, gdim, gstr, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) return fail(TBN_ERR_CUDA, "dense conv: tensor map of y failed (%d)", (int)cr);
  }
  static std::once_flag once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(once, [] {
    attr_err = cudaFuncSetAttribute(dense_conv_tc_kernel,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  });
  if (attr_err != cudaSuccess) return cuda_fail(attr_err, "cudaFuncSetAttribute(dense_conv_tc_kernel)");
  const int gy = (a.K + kFilt - 1) / kFilt;
  if (gy > 65535) return fail(TBN_ERR_UNSUPPORTED, "dense conv: grid too large");
  // persistent: one CTA per SM, shared by the filter groups
  const int gx = std::max(1, std::min(a.tiles, device_sm_count() / gy));
  dense_conv_tc_kernel<<<dim3(gx, gy), kThreads, smem, s>>>(tmap_x, tmap_y, a);
  return check_launch("dense_conv_tc_kernel");
}

}  // namespace tbn
