// tbn_conv_igemm.cu -- host dispatch of the tcgen05 implicit-GEMM two-bit
// convolution (Eq. 1, Section 2): the tile plan, the split of K for
// 1x1 layers, the space-to-depth form of a strided first layer, fused
// quantization, and the gathering modes' kernel variants.  The kernel and
// its design are in tbn_conv_igemm.cuh.
#include "tbn_conv_igemm.cuh"

namespace tbn {
namespace {

// Split K: y = 2 alpha[k] * (sum of the K ranges' partial sums, in range
// order) (+ residual), ReLU, rounded to y's dtype.  Deterministic.  Four
// consecutive outputs per thread (K % 4 == 0: 16-byte partial loads).
template <bool kVec>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ partial,
                                                           int S, int64_t mk, int K,
                                                           const float* __restrict__ alpha,
                                                           const void* residual, int relu,
                                                           void* y, int y_bf16) {
  constexpr int kV = kVec ? 4 : 1;
  const int64_t n = mk / kV;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float acc[kV];
    if constexpr (kVec) {
      float4 t = __ldg(reinterpret_cast<const float4*>(partial) + i);
      for (int s = 1; s < S; ++s) {
        const float4 u = __ldg(reinterpret_cast<const float4*>(partial + s * mk) + i);
        t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
      }
      acc[0] = t.x; acc[1] = t.y; acc[2] = t.z; acc[3] = t.w;
    } else {
      acc[0] = 0.0f;
      for (int s = 0; s < S; ++s) acc[0] += __ldg(partial + s * mk + i);
    }
    const int64_t o = i * kV;
    const int k0 = static_cast<int>(o % K);
#pragma unroll
    for (int e = 0; e < kV; ++e) {
      float v = 2.0f * __ldg(alpha + k0 + e) * acc[e];
      if (y_bf16) {
        if (residual) v += __bfloat162float(static_cast<const __nv_bfloat16*>(residual)[o + e]);
        if (relu) v = fmaxf(v, 0.0f);
        static_cast<__nv_bfloat16*>(y)[o + e] = __float2bfloat16_rn(v);
      } else {
        if (residual) v += static_cast<const float*>(residual)[o + e];
        if (relu) v = fmaxf(v, 0.0f);
        static_cast<float*>(y)[o + e] = v;
      }
    }
  }
}

// Split K within clusters: the K ranges (2 .. 8) that a cluster's CTAs take of
// each tile, with `t` set to its tiles, or 1 where the two launches of
// splitk_reduce_kernel's form are estimated to be quicker.  At most the
// p.ksplit ranges that the caller's workspace holds, and clusters in whole
// waves of those that the device runs at once (GB300: 36 of four CTAs, 15 of
// eight).  Costs in ns: a K block as in plan_cost; start, exchange and end,
// fitted, 3.5 us + 12 ns a pixel in a cluster (24 where K is no multiple of four
// and the sums go one by one); two launches 4.5 us + 12 ns a pixel + 80 ns a
// range (60), whose sums one thread adds in turn.  Measured, two launches and
// clusters: 256 x 9216 -> 4096 21.0 and 19.2 us, 256 x 4096 -> 4096 15.6 and
// 13.8, 256 x 4096 -> 1000 11.4 and 9.3 (two tiles of 128 images, six ranges), 64
// x 2048 -> 300 7.9 and 5.4; even at 64 x 25088 -> 128 (98 ranges of four K
// blocks), beyond which two launches win; 256 x 25088 -> 10 14.4 and 17.4, 64 x
// 16384 -> 10 10.0 and 12.6, 128 x 4096 -> 1001 9.5 and 10.8.
int cluster_split(const ConvProblem& p, TilePlan& t) {
  const int64_t kb = kblocks_of(p), tk = ceil_div(p.K, kBM);
  const auto block = [](int64_t bn) { return 215.0 + 0.25 * bn; };
  const bool vec = p.K % 4 == 0;
  double cost = ceil_div(kb, p.ksplit) * block(t.bn) + 4500.0 + 12.0 * t.bn + (vec ? 80.0 : 60.0) * p.ksplit;
  const int parts0 = t.tiles_n;
  int best = 1;
  for (int parts = parts0; parts <= 4 * parts0; ++parts) {
    const int bn = ceil_div(p.N, parts);
    if (ceil_div(p.N, bn) != parts) continue;
    for (int S = 2; S <= std::min(kMaxCluster, p.ksplit); ++S) {
      const int per = ceil_div(kb, S), fit = igemm_max_clusters(S);
      if ((S - 1) * per >= kb || fit < 1) continue;
      const double c = ceil_div(parts * tk, fit) * (per * block(bn) + 3500.0 + (vec ? 12.0 : 24.0) * bn);
      // narrower tiles only for a clear gain
      if (c >= (parts > t.tiles_n && best > 1 ? 0.95 : 1.0) * cost) continue;
      cost = c;
      best = S;
      t.bn = t.T = bn;
      t.tiles_n = parts;
      t.tile_n = (bn + 15) / 16 * 16;
    }
  }
  return best;
}

// Whether a layer of 64 m + 32 channels runs on tap pairs instead of pairs of
// 32-channel boxes: on the widest tiles the boxes' rows set the pace of a K
// block (256 pixels: 96 -> 256 channels, 27 x 27, 5 x 5, batch 256, 137 -> 128
// us; 160 -> 256, 3 x 3, 92.0 -> 87.7; 416 -> 384, 14 x 14, 3 x 3, 83.6 ->
// 78.5).  Narrower ones are paced by the warps' own instructions, of which the
// pairs take more (224 pixels: 224 -> 512 channels, 14 x 14, 65.5 and 65.2; 160
// -> 384, 13 x 13, 5 x 5, 77.2 and 80.8; 160 pixels: 96 -> 128, 27 x 27, 5 x
// 5, batch 32, 13.9 and 15.4).
bool tap_pairs_pay(const ConvProblem& p, const TilePlan& t) {
  return p.C > kBK && t.tile_n > 224 && p.R * p.S > 1;
}

int patch_cap_bytes(const ConvProblem& p, const TilePlan& t) {
  return tma_fed(p) ? 0 : patch_bytes_of(p, t);
}

}  // namespace

bool conv_igemm_uses_tma(const ConvProblem& p) { return use_tma(p); }

namespace {

// How the activations of a planned launch reach the ring (kMode...).
int mode_of(const ConvProblem& p, const TilePlan& t, bool s2d) {
  if (s2d) return kModeS2d;
  if (t.rowpair) return kModeRowPair;
  if (use_tma(p)) {
    if (!use_ch32(p)) return kModeTma64;
    return tap_pairs_pay(p, t) ? kModeTapPair : kModeTma32;
  }
  if (use_tma_pad(p)) return kModeTmaPad;
  return patch_cap_bytes(p, t) > 0 ? kModePatch : kModeGather;
}

// Tensor-memory columns of each resident K block (space-to-depth mode).
int resident_cols(const ConvProblem& p) {
  return p.layout == TBN_S2D_NHWC ? 8 * ceil_div(p.sh * p.sh * p.C, 16) : 0;
}

}  // namespace

// Split K when the output tiles fill fewer than half the SMs and the filter
// has at least 8 K blocks.  The tensor core's time per K block is
// proportional to the tile's pixels, but a CTA's time per K block is not
// (measured: it barely moves between 32 and 256 pixels; the operand supply
// sets it), so idle SMs are filled with K ranges of full-width tiles rather
// than with narrower tiles.
int conv_igemm_splitk(const ConvProblem& p, size_t* workspace_bytes) {
  *workspace_bytes = 0;
  // fully-connected shapes only (a 1x1 convolution over a 1x1 image): a
  // tile's pixel i is then image n0 + i, and the partial sums are stored
  // without the pixel walk of a general tile
  if (!tma_fed(p) || p.pool || p.P != 1 || p.Q != 1 || p.R != 1 || p.S != 1) return 1;
  const TilePlan t = plan_tiles(p);
  const int64_t base = static_cast<int64_t>(t.tiles_q) * t.tiles_p * t.tiles_n *
                       ((p.K + kBM - 1) / kBM);
  const int64_t kblocks = kblocks_of(p);
  const int sms = device_sm_count();
  if (2 * base > sms || kblocks < 8) return 1;
  int64_t S = std::min<int64_t>(sms / base, kblocks / 4);
  if (S < 2) return 1;
  const int64_t per = (kblocks + S - 1) / S;
  S = (kblocks + per - 1) / per;
  *workspace_bytes = static_cast<size_t>(S) * p.N * p.P * p.Q * p.K * 4;
  return static_cast<int>(S);
}

// The stride-1 convolution over the space-to-depth input that a
// TBN_S2D_NHWC problem runs as.
ConvProblem s2d_problem(const ConvProblem& p) {
  const S2dGeom g = s2d_geom(p.R, p.S, p.sh, p.P, p.Q);
  ConvProblem q = p;
  q.layout = TBN_NHWC;
  q.C = kS2dChannels;
  q.H = g.Hs;
  q.W = g.Ws;
  q.R = g.Rp;
  q.S = g.Sp;
  q.sh = q.sw = 1;
  q.ph = q.pw = 0;
  return q;
}

const char* s2d_unsupported_reason(const ConvProblem& p) {
  if (p.xdt != TBN_BF16) return "space-to-depth input must be bf16";
  if (p.sh != p.sw || p.sh < 2) return "space-to-depth needs equal strides >= 2";
  if (p.sh * p.sh * p.C > kS2dChannels) return "space-to-depth needs stride^2 * C <= 64";
  if (p.K > kBM) return "space-to-depth keeps one filter block (K <= 128) resident";
  if (p.pool || p.residual) return "space-to-depth takes no pool and no residual";
  if (p.ksplit > 1) return "space-to-depth takes no split K";
  const ConvProblem q = s2d_problem(p);
  const int64_t kb = q.R * q.S;
  if (kb > kMaxResidentKB || plan_tiles(q).tile_n + 32 * kb > kTmemCols)
    return "space-to-depth: the filter's K blocks do not fit in tensor memory beside the tile";
  return "";
}

const char* conv_igemm_unsupported_reason(const ConvProblem& p) {
  if (p.layout == TBN_S2D_NHWC) {
    const char* r = s2d_unsupported_reason(p);
    if (*r) return r;
    return conv_igemm_unsupported_reason(s2d_problem(p));
  }
  if (p.layout != TBN_NHWC) return "implicit GEMM needs NHWC";
  if (p.xdt != TBN_BF16) return "implicit GEMM needs bf16 activations";
  if (!is_aligned(p.x, 16)) return "implicit GEMM needs 16-byte aligned x";
  if (p.pool && p.residual) return "pooling with a residual is not supported";
  if (p.N > (1 << 30) || p.H > (1 << 30) || p.W > (1 << 30) || p.K > (1 << 30))
    return "dimension too large";
  if (p.C * p.R * p.S >= (int64_t(1) << 30)) return "filter too large";
  if (p.H * p.W * p.C >= (int64_t(1) << 31)) return "image too large";
  if (p.R >= (1 << 15) || p.S >= (1 << 15)) return "kernel too large";
  if (use_tma(p) && (p.ph > p.R || p.pw > p.S)) return "implicit GEMM needs pad <= kernel extent";
  const int pool_bw = pool_width(p, plan_tiles(p));
  if (pool_bw < 0 || pool_bw == 1)
    return "fused pool needs whole output rows of width 8, 16 or 32 per tile";
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return "no CUDA device";
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  if (major != 10 || minor != 3) return "implicit GEMM kernel is built for sm_103a only";
  if ((tma_fed(p) || use_tma_store(p)) && get_encode_tiled() == nullptr)
    return "cuTensorMapEncodeTiled unavailable";
  return "";
}

// A fused pool over rows of a width that the explicit implicit-GEMM algorithm
// refuses (not 8, 16 or 32) but its TMA-fed modes can pool: AUTO's choice
// then, against the CUDA-core kernel (3x3, 64 -> 128 channels, 24 x 28, batch
// 21, pooled: 454 us there).
bool conv_igemm_pools_any_width(const ConvProblem& p) {
  if (!p.pool || p.layout != TBN_NHWC || p.residual || !tma_fed(p)) return false;
  ConvProblem q = p;
  q.pool = 0;
  if (conv_igemm_unsupported_reason(q)[0] != '\0') return false;
  return pool_width(p, plan_tiles(p)) == 1;
}

int conv_igemm_mode(const ConvProblem& p0) {
  const bool s2d = p0.layout == TBN_S2D_NHWC;
  const ConvProblem p = s2d ? s2d_problem(p0) : p0;
  return mode_of(p, plan_conv(p, resident_cols(p0)), s2d);
}

tbn_status launch_conv_igemm(const ConvProblem& p0, cudaStream_t s) {
  const bool s2d = p0.layout == TBN_S2D_NHWC;
  const ConvProblem p = s2d ? s2d_problem(p0) : p0;
  const int resident = resident_cols(p0);
  TilePlan t = plan_conv(p, resident);
  const bool split = p.ksplit > 1 && p.partial != nullptr;
  const int cluster = split && is_aligned(p.partial, 16) ? cluster_split(p, t) : 1;
  IgArgs a{};
  a.N = (int)t.oN; a.C = (int)p.C; a.H = (int)p.H; a.W = (int)p.W; a.K = (int)p.K;
  a.R = (int)p.R; a.S = (int)p.S; a.sh = (int)p.sh; a.sw = (int)p.sw;
  a.ph = (int)p.ph; a.pw = (int)p.pw; a.P = (int)t.oP; a.Q = (int)t.oQ;
  a.im2col = t.im2col ? 1 : 0; a.iP = (int)p.P; a.iQ = (int)p.Q;
  if (t.rowpair) {   // the convolution of the row pairs
    a.iP /= 2;
    a.sh = 2;
    a.R += 1;
  }
  a.bw = t.bw; a.bh = t.bh; a.bn = t.bn; a.tile_n = t.tile_n;
  a.tiles_q = t.tiles_q; a.tiles_p = t.tiles_p;
  a.tiles_k = ceil_div(p.K, kBM);
  const int64_t tiles = static_cast<int64_t>(t.tiles_q) * t.tiles_p * t.tiles_n * a.tiles_k;
  a.ncodes = (int)(p.C * p.R * p.S);
  a.kblocks = t.rowpair ? a.R * a.S * a.C / kBK : static_cast<int>(kblocks_of(p));
  a.cluster = cluster > 1 ? 1 : 0;
  a.ksplit = a.cluster ? cluster : split ? p.ksplit : 1;
  a.kb_per = ceil_div(a.kblocks, a.ksplit);
  if (split && (!tma_fed(p) || p.pool || p.P != 1 || p.Q != 1 || p.R != 1 || p.S != 1 ||
                (a.ksplit - 1) * a.kb_per >= a.kblocks))
    return fail(TBN_ERR_INVALID_ARG, "implicit GEMM: bad split-K request");
  if (tiles * a.ksplit > 0x7fffffffLL) return fail(TBN_ERR_UNSUPPORTED, "implicit GEMM: too many tiles");
  a.base_tiles = static_cast<int>(tiles);
  a.tiles = static_cast<int>(tiles * a.ksplit);
  a.partial = split ? p.partial : nullptr;
  a.by_base = fast_div(a.cluster ? a.ksplit : a.base_tiles);
  a.by_k = fast_div(a.tiles_k);
  a.by_tq = fast_div(a.tiles_q);
  a.by_tp = fast_div(a.tiles_p);
  a.by_iq = fast_div(a.iQ);
  a.by_ip = fast_div(a.iP);
  a.wpf = (a.ncodes + 15) / 16;
  if (s2d) {
    // codes of the original (r, s, c) filter
    a.wpf = static_cast<int>((p0.C * p0.R * p0.S + 15) / 16);
    a.s2d_s = static_cast<int>(p0.sh);
    a.s2d_C = static_cast<int>(p0.C);
    a.s2d_R = static_cast<int>(p0.R);
    a.s2d_S = static_cast<int>(p0.S);
    if (split || a.tiles_k != 1 || a.kblocks > kMaxResidentKB ||
        t.tile_n + resident * a.kblocks > kTmemCols || p.pool || p.residual)
      return fail(TBN_ERR_UNSUPPORTED, "implicit GEMM: space-to-depth problem out of range");
  }
  // tiles of at most 176 pixels: two accumulators, so each tile's MMAs
  // overlap the previous tile's epilogue (space-to-depth mode keeps its
  // resident K blocks where the second accumulator would be)
  a.acc2 = (!s2d && t.tile_n <= kAcc2Cols) ? 1 : 0;
  a.x = static_cast<const __nv_bfloat16*>(p.x);
  a.codes = p.codes; a.alpha = p.alpha; a.y = p.y; a.residual = p.residual;
  if (p0.wq != nullptr) {
    if (s2d || split || !use_tma(p) || a.wpf > 2048 || p0.gbar == nullptr)
      return fail(TBN_ERR_UNSUPPORTED,
                  "implicit GEMM: fused quantization needs TMA activations (C %% 32 == 0, "
                  "stride <= 2), at most 2048 words per filter and no split of K");
    a.wq = p0.wq;
    a.codes_w = const_cast<uint32_t*>(p0.codes);
    a.alpha_w = const_cast<float*>(p0.alpha);
    a.gbar = p0.gbar;
    a.wq_vec = (is_aligned(p0.wq, 16) && a.ncodes % 4 == 0) ? 1 : 0;
  }
  a.relu = p.relu; a.y_bf16 = p.ydt == TBN_BF16 ? 1 : 0;
  a.err = device_error_word();
  const int pw = pool_width(p, t);
  const bool tst = use_tma_store(p) && !split;   // partial sums: direct fp32 stores
  if (split) {
    // the K ranges' partial sums, then (unless each cluster adds its own)
    // their ordered sum with the epilogue
    const tbn_status st = use_tma_pad(p) ? launch_igemm_pad(p, t, a, pw, false, s)
                          : use_ch32(p)  ? launch_igemm_tma32(p, t, a, pw, false, false, s)
                                         : launch_igemm_tma64(p, t, a, pw, false, false, s);
    if (st != TBN_OK || a.cluster) return st;
    const int64_t mk = p.N * p.P * p.Q * p.K;
    const bool vec = p.K % 4 == 0 && is_aligned(p.partial, 16);
    const int64_t items = vec ? mk / 4 : mk;
    const int64_t blocks = std::min<int64_t>((items + 255) / 256, int64_t(device_sm_count()) * 16);
    if (vec)
      splitk_reduce_kernel<true><<<static_cast<unsigned>(blocks), 256, 0, s>>>(
          p.partial, a.ksplit, mk, (int)p.K, p.alpha, p.residual, p.relu, p.y,
          p.ydt == TBN_BF16 ? 1 : 0);
    else
      splitk_reduce_kernel<false><<<static_cast<unsigned>(blocks), 256, 0, s>>>(
          p.partial, a.ksplit, mk, (int)p.K, p.alpha, p.residual, p.relu, p.y,
          p.ydt == TBN_BF16 ? 1 : 0);
    return check_launch("splitk_reduce_kernel");
  }
  const bool fuse = a.wq != nullptr;
  switch (mode_of(p, t, s2d)) {
    case kModeS2d:
      return tst ? launch_t<kModeS2d, 0, true, false>(p, t, a, s)
                 : launch_t<kModeS2d, 0, false, false>(p, t, a, s);
    case kModeRowPair: return launch_igemm_rowpair(p, t, a, s);
    case kModeTapPair: return launch_igemm_tappair(p, t, a, pw, tst, fuse, s);
    case kModeTma32: return launch_igemm_tma32(p, t, a, pw, tst, fuse, s);
    case kModeTma64: return launch_igemm_tma64(p, t, a, pw, tst, fuse, s);
    case kModeTmaPad: return launch_igemm_pad(p, t, a, pw, tst, s);
    case kModePatch:
      a.PR = (t.bh - 1) * a.sh + a.R;
      a.PW = a.W + 2 * a.pw;
      a.patch_cap = patch_cap_bytes(p, t);
      a.patch_bulk = a.pw == 0 ? 1 : 0;
      a.x_bytes = static_cast<long long>(p.N) * p.H * p.W * p.C * 2;
      return tst ? launch_pool<kModePatch, true, false>(p, t, a, pw, s)
                 : launch_pool<kModePatch, false, false>(p, t, a, pw, s);
  }
  return tst ? launch_pool<kModeGather, true, false>(p, t, a, pw, s)
             : launch_pool<kModeGather, false, false>(p, t, a, pw, s);
}

}  // namespace tbn
