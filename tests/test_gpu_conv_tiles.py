"""GPU parity of the implicit GEMM's tile shapes and epilogues against the
oracle's convolution, at the sizes where a tile, a box of filters or a
column group begins or ends.  Tolerances as in parity_util."""
import pytest
import torch

import oracle
import paper_1701_00485_gb300 as tbn
from paper_1701_00485_gb300 import inputs
from parity_util import ConvCase, assert_within, device_us, random_sites

pytestmark = pytest.mark.gpu


def _case(N, C, H, W, K, R, S, stride, pad, seed):
    g = inputs.generator(seed)
    x = torch.randn(N, C, H, W, generator=g)
    return ConvCase(x, inputs.normal((K, C, R, S), 1.2, g), stride, pad)


@pytest.mark.parametrize("K", [8, 64, 72, 136])
@pytest.mark.parametrize("N,hw", [(1, 3), (2, 7), (3, 16)])
def test_residual_epilogue_filter_boxes(K, N, hw):
    """The residual joins in the fragment epilogue: one and two 64-filter
    boxes, ragged ones, and pixel counts off the 32-column groups."""
    c = _case(N, 64, hw, hw, K, 3, 3, (1, 1), (1, 1), seed=100 * K + hw)
    y_orc, bound = c.oracle_full(torch.bfloat16)
    res = torch.randn(*y_orc.shape, generator=inputs.generator(K)).to(torch.bfloat16)
    for relu in (False, True):
        want = oracle.epilogue(y_orc, res.float().numpy(), relu=relu)
        y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.bfloat16,
                      algo=tbn.TBN_CONV_IMPLICIT_GEMM, relu=relu, residual=res)
        assert_within(y, want, bound, out_bf16=True, epilogue=True,
                      what="residual K=%d N=%d %d" % (K, N, hw))


RUNS = [
    # N, C, H, W, K, R, S, stride, pad: inputs of at least 128 KiB, whose
    # tiles are runs of pixels that cross rows and images
    (9, 64, 13, 13, 136, 3, 3, (1, 1), (1, 1)),
    (5, 64, 23, 21, 72, 3, 3, (2, 2), (1, 1)),      # odd sizes, stride 2
    (3, 96, 27, 29, 64, 5, 5, (1, 1), (2, 2)),      # 32-channel boxes, ragged last block
    (7, 128, 15, 15, 128, 1, 1, (2, 2), (0, 0)),    # projection shortcut
    (3, 64, 40, 30, 40, 2, 3, (1, 2), (1, 0)),      # R != S, stride and pad differ by axis
    (2, 128, 3, 300, 128, 3, 3, (1, 1), (1, 1)),    # rows longer than a tile
    (300, 64, 2, 2, 64, 3, 3, (1, 1), (1, 1)),      # a tile holds many images
]


@pytest.mark.parametrize("case", RUNS)
def test_pixel_run_tiles(case):
    c = _case(*case, seed=sum(case[:7]))
    y_orc, bound = c.oracle_full(torch.bfloat16)
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.float32,
                  algo=tbn.TBN_CONV_IMPLICIT_GEMM)
    assert_within(y, y_orc, bound, out_bf16=False, what="runs %s" % (case,))
    res = torch.randn(*y_orc.shape, generator=inputs.generator(3)).to(torch.bfloat16)
    want = oracle.epilogue(y_orc, res.float().numpy(), relu=True)
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.bfloat16,
                  algo=tbn.TBN_CONV_IMPLICIT_GEMM, relu=True, residual=res)
    assert_within(y, want, bound, out_bf16=True, epilogue=True, what="runs epi %s" % (case,))


@pytest.mark.parametrize("N,C,hw", [(5, 128, 16), (21, 64, 8), (3, 96, 32)])
def test_pixel_run_tiles_pooled(N, C, hw):
    """Fused 2x2 pool over runs of row pairs that cross images."""
    c = _case(N, C, hw, hw, 72, 3, 3, (1, 1), (1, 1), seed=N)
    y_orc, bound = c.oracle_full(torch.bfloat16)
    want = oracle.maxpool2d_nchw(oracle.epilogue(y_orc, None, relu=True), (2, 2), (2, 2))
    P = hw // 2
    bound = bound.reshape(N, 72, P, 2, P, 2).max(axis=(3, 5))
    Wl, codes, alpha = c.quantize_gpu(tbn.TBN_NHWC)
    x = c.x.to(torch.bfloat16).permute(0, 2, 3, 1).contiguous().cuda()
    for dt in (torch.float32, torch.bfloat16):
        y = tbn.tbn_conv2d_fwd(x, codes, alpha, 72, 3, 3, (1, 1), (1, 1), out_dtype=dt, relu=True,
                               pool=2, algo=tbn.TBN_CONV_IMPLICIT_GEMM)
        y = y.float().cpu().permute(0, 3, 1, 2).numpy()
        assert_within(y, want, bound, out_bf16=dt == torch.bfloat16, epilogue=True,
                      what="pooled runs %d %d" % (N, hw))


PADDED = [
    # N, C, H, W, K, R, S, stride, pad: C % 8 == 0, no multiple of 32: each
    # tap's last 64-channel box reaches past C
    (3, 8, 12, 11, 40, 3, 3, (1, 1), (1, 1)),       # one step per K block, half-word taps
    (9, 40, 27, 27, 136, 5, 5, (1, 1), (2, 2)),     # runs of pixels, two filter tiles
    (2, 72, 9, 10, 72, 3, 3, (2, 2), (1, 1)),       # a block of 8 channels after one of 64
    (5, 120, 14, 13, 64, 1, 1, (1, 1), (0, 0)),     # 1x1, half a word at the row's end
    (1, 48, 3, 300, 24, 2, 3, (1, 2), (1, 0)),      # whole words, columns split
    (130, 200, 1, 1, 300, 1, 1, (1, 1), (0, 0)),    # a linear layer's shape
]


@pytest.mark.parametrize("case", PADDED)
def test_padded_channel_blocks(case):
    assert tbn._conv_mode(*case) == "pad"
    c = _case(*case, seed=sum(case[:7]))
    y_orc, bound = c.oracle_full(torch.bfloat16)
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.float32,
                  algo=tbn.TBN_CONV_IMPLICIT_GEMM)
    assert_within(y, y_orc, bound, out_bf16=False, what="padded %s" % (case,))
    for dt in (torch.float32, torch.bfloat16):
        res = torch.randn(*y_orc.shape, generator=inputs.generator(3)).to(dt)
        want = oracle.epilogue(y_orc, res.float().numpy(), relu=True)
        y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, dt, algo=tbn.TBN_CONV_IMPLICIT_GEMM, relu=True,
                      residual=res)
        assert_within(y, want, bound, out_bf16=dt == torch.bfloat16, epilogue=True,
                      what="padded epi %s" % (case,))


FEW_CHANNELS = [
    # few channels under large filters: the modes whose threads build the operand
    (64, 8, 32, 31, 40, 7, 7, (1, 1), (3, 3), "patch"),
    (64, 24, 30, 32, 72, 9, 9, (1, 1), (4, 4), "gather"),
    (2, 8, 45, 50, 16, 11, 11, (2, 2), (5, 5), "patch"),
    (8, 8, 40, 36, 40, 7, 7, (1, 1), (3, 3), "pad"),    # one wave: boxes cut finer
]


@pytest.mark.parametrize("case", FEW_CHANNELS)
def test_few_channels(case):
    *case, mode = case
    assert tbn._conv_mode(*case) == mode
    c = _case(*case, seed=sum(case[:7]))
    y_orc, bound = c.oracle_full(torch.bfloat16)
    for dt in (torch.float32, torch.bfloat16):
        y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, dt)
        assert_within(y, y_orc, bound, out_bf16=dt == torch.bfloat16,
                      what="few channels %s" % (case,))
    assert tbn.tbn_device_error() == 0


@pytest.mark.parametrize("R", [7, 11])
def test_few_channels_cost_no_more_than_more(R):
    """A K block holds eight taps of 8 channels; a box of each tap's own would
    make such layers slower than those of 16 channels."""
    us = {}
    for C in (8, 16):
        g = inputs.generator(C)
        x = torch.randn(64, 32, 32, C, generator=g).to(torch.bfloat16).cuda()
        codes, alpha = tbn.tbn_quantize_pack(inputs.normal((64, R * R * C), 1.2, g).cuda())
        out = torch.empty(64, 32, 32, 64, dtype=torch.bfloat16, device="cuda")
        us[C] = device_us(lambda: tbn.tbn_conv2d_fwd(x, codes, alpha, 64, R, R, (1, 1),
                                                     (R // 2, R // 2), out=out))
    assert us[8] <= 1.3 * us[16], us


def test_direct_stores_without_a_residual_cost_less_than_with_one():
    """Outputs that no TMA store takes, stored by a gathering mode: what the
    residual's requests ahead keep in registers is not paid without one."""
    g = inputs.generator(65)
    x = torch.randn(64, 32, 32, 12, generator=g).to(torch.bfloat16).cuda()
    codes, alpha = tbn.tbn_quantize_pack(inputs.normal((33, 9 * 12), 1.2, g).cuda())
    out = torch.empty(64, 32, 32, 33, device="cuda")
    res = torch.randn(64, 32, 32, 33, generator=g).cuda()
    us = [device_us(lambda: tbn.tbn_conv2d_fwd(x, codes, alpha, 33, 3, 3, (1, 1), (1, 1), out=out,
                                               out_dtype=torch.float32, residual=r))
          for r in (None, res)]
    assert us[0] <= 0.8 * us[1], us


@pytest.mark.parametrize("B,K_in,K_out", [(9, 1000, 70), (64, 2008, 130), (2, 520, 33)])
def test_padded_linear(B, K_in, K_out):
    """Fully-connected layers whose K_in is a multiple of 8 only, with the
    workspace that lets K be split."""
    g = inputs.generator(K_in)
    x = torch.randn(B, K_in, generator=g).to(torch.bfloat16)
    W = torch.randn(K_out, K_in, generator=g)
    codes, alpha = tbn.tbn_quantize_pack(W.cuda())
    n = tbn.tbn_linear_workspace_bytes(B, K_in, K_out)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda") if n else None
    wt, al = oracle.quantize(W.numpy())
    want, bound = oracle.linear(x.float().numpy(), wt, al)
    for w in {None, ws}:
        y = tbn.tbn_linear_fwd_ws(x.cuda(), codes, alpha, K_out, w, out_dtype=torch.float32)
        assert_within(y.cpu().numpy(), want, bound, out_bf16=False, what="padded linear")


@pytest.mark.parametrize("case,pool", [
    ((8, 96, 8, 8, 130, 3, 3, (1, 1), (1, 1)), 0),    # nine taps: the last has no partner
    ((8, 96, 8, 8, 64, 3, 3, (1, 1), (1, 1)), 2),
    ((4, 160, 8, 7, 72, 1, 2, (1, 1), (0, 1)), 0),    # one pair, two whole blocks a tap
    ((8, 160, 7, 7, 40, 2, 4, (1, 1), (1, 2)), 0),    # pairs that end in the next row
    ((4, 96, 15, 8, 24, 5, 5, (2, 1), (2, 2)), 0),   # strided
    ((2, 224, 8, 16, 24, 3, 1, (1, 1), (1, 0)), 0),
    ((256, 96, 27, 27, 256, 5, 5, (1, 1), (2, 2)), 0),   # runs of pixels
])
def test_tap_pairs(case, pool):
    """64 m + 32 channels on tiles of 256 pixels: K blocks of tap pairs."""
    c = _case(*case, seed=sum(case[:7]))
    N, C, H, W, K, R, S, st, pad = case
    Wl, codes, alpha = c.quantize_gpu(tbn.TBN_NHWC)
    x = c.x.to(torch.bfloat16).permute(0, 2, 3, 1).contiguous().cuda()
    for dt in (torch.float32, torch.bfloat16):
        assert tbn._conv_mode(*case, out_dtype=dt, pool=pool) == "tappair"
        y = tbn.tbn_conv2d_fwd(x, codes, alpha, K, R, S, st, pad, out_dtype=dt, relu=bool(pool),
                               pool=pool)
        assert tbn.tbn_device_error() == 0
        got = y.float().cpu().permute(0, 3, 1, 2).contiguous().numpy()
        if N > 64:
            sites = random_sites(got.shape, 2000, seed=5)
            want, bound = c.oracle_sites(torch.bfloat16, sites)
            got = got[tuple(sites.T)]
        else:
            want, bound = c.oracle_full(torch.bfloat16)
            if pool:
                P, Q = want.shape[2] // 2, want.shape[3] // 2
                want = oracle.maxpool2d_nchw(oracle.epilogue(want, None, relu=True), (2, 2), (2, 2))
                bound = bound[:, :, :2 * P, :2 * Q].reshape(N, K, P, 2, Q, 2).max(axis=(3, 5))
        assert_within(got, want, bound, out_bf16=dt == torch.bfloat16, epilogue=bool(pool),
                      what="tap pairs %s" % (case,))


@pytest.mark.parametrize("B,K_in,K_out,dtype,res", [
    (256, 4096, 1000, torch.bfloat16, False),   # tiles of 128 images
    (300, 4096, 512, torch.float32, True),      # a last tile of fewer images
    (33, 2016, 131, torch.bfloat16, True),      # K_out odd, 32-channel boxes, a ragged last range
    (9, 520, 128, torch.float32, False),        # two ranges, padded channels
    (17, 8192, 129, torch.bfloat16, False),     # eight ranges, one filter in the last tile
    (64, 100352, 64, torch.float32, False),     # a filter so long that it takes two launches
])
def test_linear_split_in_clusters(B, K_in, K_out, dtype, res):
    """Split K whose ranges are added by the clusters that computed them, y at
    an odd element offset and aligned."""
    g = inputs.generator(B + K_in)
    x = torch.randn(B, K_in, generator=g).to(torch.bfloat16)
    W = torch.randn(K_out, K_in, generator=g)
    r = torch.randn(B, K_out, generator=g).to(dtype) if res else None
    codes, alpha = tbn.tbn_quantize_pack(W.cuda())
    n = tbn.tbn_linear_workspace_bytes(B, K_in, K_out)
    assert n >= 2 * 4 * B * K_out
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
    wt, al = oracle.quantize(W.numpy())
    y_orc, bound = oracle.linear(x.float().numpy(), wt, al)
    want = oracle.epilogue(y_orc, r.float().numpy() if res else None, relu=True)
    for off in (0, 1):
        buf = torch.full((B * K_out + 2,), float("nan"), dtype=dtype, device="cuda")
        y = buf[off:off + B * K_out].view(B, K_out)
        tbn.tbn_linear_fwd_ws(x.cuda(), codes, alpha, K_out, ws, relu=True,
                              residual=r.cuda() if res else None, out=y, out_dtype=dtype)
        assert_within(y.float().cpu().numpy(), want, bound, out_bf16=dtype == torch.bfloat16,
                      epilogue=True, what="clusters %s" % ((B, K_in, K_out, off),))
        assert torch.isnan(buf[:off]).all() and torch.isnan(buf[off + B * K_out:]).all()
    assert tbn.tbn_device_error() == 0


def test_linear_split_of_many_ranges_and_few_outputs():
    """Very long filters and a count of outputs that is no multiple of four: the
    two launches, whose many ranges a cluster's eight cannot match."""
    us = {}
    for K_out in (10, 12):
        x = torch.randn(64, 16384, device="cuda").to(torch.bfloat16)
        codes, alpha = tbn.tbn_quantize_pack(torch.randn(K_out, 16384, device="cuda"))
        ws = torch.empty(tbn.tbn_linear_workspace_bytes(64, 16384, K_out), dtype=torch.uint8,
                         device="cuda")
        out = torch.empty(64, K_out, dtype=torch.bfloat16, device="cuda")
        us[K_out] = device_us(lambda: tbn.tbn_linear_fwd_ws(x, codes, alpha, K_out, ws, out=out))
    assert us[10] <= 0.92 * us[12], us


@pytest.mark.parametrize("case", [
    (3, 64, 28, 28, 72, 3, 3, (1, 1), (1, 1)),      # even map: runs of row pairs
    (2, 64, 13, 11, 136, 3, 3, (1, 1), (1, 1)),     # odd: the last row and column drop
    (7, 64, 7, 9, 64, 3, 3, (1, 1), (1, 1)),        # several images per tile, odd rows
    (2, 40, 20, 24, 64, 3, 3, (1, 1), (1, 1)),      # padded channels
    (1, 96, 34, 128, 24, 3, 3, (1, 1), (1, 1)),     # the widest rows that pair up
    (2, 64, 45, 44, 64, 3, 3, (2, 2), (1, 1)),      # strided
])
def test_pool_of_any_width(case):
    """AUTO pools rows of other widths than 8, 16 and 32 in the implicit
    GEMM; naming that algorithm is refused as before."""
    c = _case(*case, seed=sum(case[:7]))
    K = case[4]
    y_orc, bound = c.oracle_full(torch.bfloat16)
    P, Q = y_orc.shape[2] // 2, y_orc.shape[3] // 2
    want = oracle.maxpool2d_nchw(oracle.epilogue(y_orc, None, relu=True), (2, 2), (2, 2))
    bound = bound[:, :, :2 * P, :2 * Q].reshape(-1, K, P, 2, Q, 2).max(axis=(3, 5))
    Wl, codes, alpha = c.quantize_gpu(tbn.TBN_NHWC)
    x = c.x.to(torch.bfloat16).permute(0, 2, 3, 1).contiguous().cuda()
    args = (x, codes, alpha, K, case[5], case[6], case[7], case[8])
    for dt in (torch.float32, torch.bfloat16):
        y = tbn.tbn_conv2d_fwd(*args, out_dtype=dt, relu=True, pool=2)
        y = y.float().cpu().permute(0, 3, 1, 2).numpy()
        assert_within(y, want, bound, out_bf16=dt == torch.bfloat16, epilogue=True,
                      what="any width %s" % (case,))
    assert tbn.tbn_device_error() == 0
    with pytest.raises(tbn.TBNError):
        tbn.tbn_conv2d_fwd(*args, relu=True, pool=2, algo=tbn.TBN_CONV_IMPLICIT_GEMM)


FEW_FILTERS = [
    # at most 64 filters and an even number of output rows, but work for one wave
    # of tiles only: runs of pixels
    (6, 64, 56, 56, 64, 3, 3, (1, 1), (1, 1)),
    (9, 128, 14, 17, 40, 3, 3, (1, 1), (1, 1)),     # ragged filters, odd width
    (5, 64, 21, 24, 8, 2, 3, (1, 2), (0, 1)),       # R = 2, column stride 2
    (3, 64, 18, 60, 64, 5, 5, (1, 1), (2, 2)),
]


@pytest.mark.parametrize("case", FEW_FILTERS)
def test_few_filters(case):
    assert tbn._conv_mode(*case) == "tma64"
    _check_staged_outputs(case, "few filters")


def _check_staged_outputs(case, what):
    c = _case(*case, seed=sum(case[:7]))
    y_orc, bound = c.oracle_full(torch.bfloat16)
    assert y_orc.shape[2] % 2 == 0
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.bfloat16)
    assert_within(y, y_orc, bound, out_bf16=True, what="%s %s" % (what, case))
    res = torch.randn(*y_orc.shape, generator=inputs.generator(3)).to(torch.bfloat16)
    want = oracle.epilogue(y_orc, res.float().numpy(), relu=True)
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.bfloat16, relu=True, residual=res)
    assert_within(y, want, bound, out_bf16=True, epilogue=True, what="%s epi %s" % (what, case))


ROW_PAIRS = [
    # N, C, H, W, K, R, S, stride, pad: at most 64 filters, an even number of
    # output rows, and work for two waves of tiles, so that pairs pay
    (64, 64, 28, 28, 64, 3, 3, (1, 1), (1, 1)),     # 64 filters, several tiles per CTA
    (64, 128, 28, 27, 40, 3, 3, (1, 1), (1, 1)),    # ragged filters, odd width, 128 channels
    (48, 64, 33, 56, 8, 2, 3, (1, 2), (0, 1)),      # R = 2, column stride 2
    (64, 64, 30, 31, 56, 5, 5, (1, 1), (2, 2)),
    (90, 64, 41, 27, 64, 2, 2, (1, 1), (0, 0)),     # no padding
    (300, 64, 12, 28, 24, 3, 3, (1, 2), (1, 1)),    # a tile holds two images
]


@pytest.mark.parametrize("case", ROW_PAIRS)
def test_row_pairs(case):
    for residual in (False, True):
        assert tbn._conv_mode(*case, residual=residual) == "rowpair"
    _check_staged_outputs(case, "row pairs")


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("case,mode", [
    ((64, 64, 28, 28, 48, 3, 3, (1, 1), (1, 1)), "rowpair"),
    ((48, 64, 33, 56, 8, 2, 3, (1, 2), (0, 1)), "rowpair"),
    ((64, 64, 30, 31, 56, 5, 5, (1, 1), (2, 2)), "rowpair"),
    ((34, 64, 16, 16, 48, 3, 3, (1, 1), (1, 1)), "tma64"),
])
def test_row_pairs_not_finite(case, mode, value):
    """An infinite or NaN input reaches the outputs whose taps read it and no
    others, although both rows of a pair are computed from the same boxes."""
    assert tbn._conv_mode(*case) == mode
    N, C, H, W, K, R, S, st, pd = case
    g = inputs.generator(11)
    x = torch.randn(N, C, H, W, generator=g)
    x[2, 5, 7, 9] = value       # an odd row: the first tap row of one pair, the last of another
    x[4, 60, 0, 0] = value
    x[33, 1, 14, W - 1] = value
    x[N - 1, 63, H - 1, 3] = value
    c = ConvCase(x, inputs.normal((K, C, R, S), 1.2, g), st, pd)
    y = c.run_gpu(tbn.TBN_NHWC, torch.bfloat16, torch.bfloat16)
    assert tbn.tbn_device_error() == 0
    wt, al = oracle.quantize(c.W.reshape(K, -1).numpy())
    w = torch.from_numpy((wt * al[:, None]).reshape(c.W.shape))
    ref = torch.nn.functional.conv2d(x.to(torch.bfloat16).double(), w.double(), stride=st,
                                     padding=pd).numpy()
    fin = torch.isfinite(torch.from_numpy(ref)).numpy()
    assert K * 4 <= (~fin).sum() <= K * 4 * R * S
    assert (torch.isnan(torch.from_numpy(y)).numpy() == torch.isnan(torch.from_numpy(ref)).numpy()).all()
    inf = ~fin & ~torch.isnan(torch.from_numpy(ref)).numpy()
    assert (y[inf] == ref[inf]).all()
    assert (abs(y[fin] - ref[fin]) <= 2.0 ** -7 * abs(ref[fin]) + 1e-3).all()


def test_row_pairs_cost_the_same_for_any_input():
    """A batch of NaN (a diverged network) takes no longer than another."""
    g = inputs.generator(12)
    codes, alpha = tbn.tbn_quantize_pack(inputs.normal((64, 576), 1.2, g).cuda())
    x = torch.randn(64, 56, 56, 64, generator=g).to(torch.bfloat16).cuda()
    out = torch.empty_like(x)
    us = {}
    for name, xs in (("finite", x), ("nan", torch.full_like(x, float("nan"))),
                     ("inf", torch.full_like(x, float("inf")))):
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                tbn.tbn_conv2d_fwd(xs, codes, alpha, 64, 3, 3, (1, 1), (1, 1), out=out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 100.0)
        us[name] = best
        assert tbn.tbn_device_error() == 0
        if name == "nan":
            assert torch.isnan(out).all()
    # some 25 us each; ten times that is far beyond any noise, and far below a
    # recomputation of such sums (milliseconds)
    assert max(us["nan"], us["inf"]) <= 10.0 * us["finite"], us
