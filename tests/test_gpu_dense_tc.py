"""The tensor-core form of the full-precision first convolution (fp32 weights
as three bf16 terms) against the oracle, at the edges of its tiles, filter
groups and weight blocks, and with infinities and NaN.

Tolerance: the products are exact and at most n = C*R*S sums of each of the
three terms round in fp32, so |err| <= n * 2^-24 * sum|x w| as for the
CUDA-core kernel, plus the bf16 rounding of the output."""
import numpy as np
import pytest
import torch

import oracle
import paper_1701_00485_gb300 as tbn
from paper_1701_00485_gb300 import inputs
from parity_util import device_us

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, R, S, stride, pad
    (2, 3, 32, 32, 64, 7, 7, (2, 2), (3, 3)),     # two whole tiles per image
    (3, 3, 30, 40, 72, 7, 7, (2, 2), (3, 3)),     # ragged last tile, second filter group
    (1, 1, 8, 8, 8, 3, 3, (2, 2), (1, 1)),        # one partial tile, one block
    (2, 4, 16, 24, 16, 5, 8, (1, 2), (0, 0)),     # 8 taps, even padding, row stride 1
    (1, 5, 33, 64, 64, 8, 4, (4, 4), (2, 1)),     # all five weight blocks
    (200, 3, 16, 16, 64, 7, 7, (2, 2), (3, 3)),   # several tiles per CTA
    (1, 3, 9, 224, 8, 7, 7, (2, 2), (3, 3)),      # the widest rows of the workload
]


def _run(x, w, st, pd, relu=False):
    y = tbn.tbn_dense_conv2d_fwd(x.cuda(), w.cuda(), st, pd, layout=tbn.TBN_NCHW_NHWC,
                                 out_dtype=torch.bfloat16, relu=relu)
    torch.cuda.synchronize()
    assert tbn.tbn_device_error() == 0
    return y.float().cpu().permute(0, 3, 1, 2).numpy()


@pytest.mark.parametrize("case", CASES)
def test_dense_tc_matches_oracle(case):
    N, C, H, W, K, R, S, st, pd = case
    g = inputs.generator(sum(case[:7]))
    x = torch.randn(N, C, H, W, generator=g).to(torch.bfloat16)
    w = inputs.he_normal(K, C, R, S, g)
    want, bound = oracle.dense_conv2d_nchw(x.float().numpy(), w.numpy(), st, pd)
    for relu in (False, True):
        ref = np.maximum(want, 0.0) if relu else want
        err = np.abs(_run(x, w, st, pd, relu).astype(np.float64) - ref)
        tol = C * R * S * 2.0 ** -24 * bound + 2.0 ** -8 * np.abs(ref)
        assert np.all(err <= tol), float(np.max(err - tol))


def test_dense_tc_single_products():
    """One tap, 24-bit weights: each output is a single product rounded once to
    bf16, at most half an ulp away."""
    g = inputs.generator(9)
    x = torch.ones(1, 1, 8, 8, dtype=torch.bfloat16)
    w = (torch.rand(64, 1, 1, 1, generator=g) + 1) * (1 + 2.0 ** -23)
    y = _run(x, w, (1, 2), (0, 0))
    want = w.reshape(1, 64, 1, 1).double().numpy() * np.ones(y.shape)
    assert np.array_equal(y, torch.from_numpy(want).to(torch.bfloat16).float().numpy())


def test_dense_tc_weight_terms():
    """Weights that need all three terms: two taps cancel to a few units of the
    24th bit, which the result holds exactly; without the third term, or with it
    in the wrong place, it is 0 or a multiple of 2^-15."""
    g = inputs.generator(9)
    x = torch.ones(1, 1, 8, 8, dtype=torch.bfloat16)
    x[..., 1::2] = -1.0
    w0 = torch.randint(1 << 23, (1 << 24) - 8, (64,), generator=g)   # 24 bits, [1, 2)
    d = torch.randint(1, 8, (64,), generator=g)
    w = torch.stack((w0 + d, w0), 1).float().reshape(64, 1, 1, 2) * 2.0 ** -23
    assert torch.equal(w.double() * 2.0 ** 23, torch.stack((w0 + d, w0), 1).reshape(w.shape).double())
    y = _run(x, w, (1, 2), (0, 0))
    want = (d.double() * 2.0 ** -23).reshape(1, 64, 1, 1).numpy() * np.ones(y.shape)
    assert np.array_equal(y.astype(np.float64), want)


@pytest.mark.parametrize("case", [
    (8, 3, 64, 64, 7, 7, (2, 2), (3, 3)),     # the stem's filter, three weight blocks and two more
    (8, 1, 64, 64, 3, 3, (2, 2), (1, 1)),
    (8, 4, 64, 64, 5, 7, (2, 2), (2, 3)),
])
def test_dense_tc_sums_in_fp32(case):
    """The sums' own error: two further channels, one tap each, take the exact
    result away from the first filter's outputs (rounded to bf16, then what that
    leaves), so what remains is the rounding of the sums, and the output's bf16
    hides none of it.  At most n additions of half a unit of sum|x w| each; the
    rms is below that of fp32 sums tap by tap."""
    N, C, H, W, R, S, st, pd = case
    g = inputs.generator(sum(case[:6]))
    x = torch.randn(N, C, H, W, generator=g).to(torch.bfloat16)
    w = inputs.he_normal(8, C, R, S, g)
    conv = torch.nn.functional.conv2d
    ref = conv(x.double(), w[:1].double(), stride=st, padding=pd)[:, 0]
    mag = conv(x.double().abs(), w[:1].double().abs(), stride=st, padding=pd)[:, 0].numpy()
    P, Q = ref.shape[1:]
    xe = torch.zeros(N, C + 2, H, W, dtype=torch.bfloat16)
    xe[:, :C] = x
    left = ref
    for i in range(2):
        xe[:, C + i, :P * st[0]:st[0], :Q * st[1]:st[1]] = (-left).to(torch.bfloat16)
        left = left + (-left).to(torch.bfloat16).double()
    we = torch.zeros(8, C + 2, R, S)
    we[:, :C] = w
    we[:, C:, pd[0], pd[1]] = 1.0
    err = {}
    for dt in (torch.bfloat16, torch.float32):    # tensor cores; CUDA cores, tap by tap
        y = tbn.tbn_dense_conv2d_fwd(xe.cuda(), we.cuda(), st, pd, layout=tbn.TBN_NCHW_NHWC,
                                     out_dtype=dt)
        torch.cuda.synchronize()
        err[dt] = (y[..., 0].double().cpu() - left).numpy()
    e = err[torch.bfloat16]
    assert np.all(np.abs(e) <= C * R * S * 2.0 ** -24 * mag + 2.0 ** -8 * np.abs(left.numpy()))
    rms = {dt: float(np.sqrt(np.mean(v ** 2))) for dt, v in err.items()}
    assert rms[torch.bfloat16] <= rms[torch.float32], rms


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.3e38])
def test_dense_tc_not_finite(value):
    """An infinite, NaN or overflowing input touches the outputs whose taps
    read it, as in fp32 arithmetic, and no other."""
    g = inputs.generator(4)
    x = torch.randn(2, 3, 24, 24, generator=g)
    x[0, 1, 7, 9] = value
    x = x.to(torch.bfloat16)
    w = inputs.he_normal(16, 3, 7, 7, g)
    y = _run(x, w, (2, 2), (3, 3))
    ref = torch.nn.functional.conv2d(x.double(), w.double(), stride=2, padding=3)
    ref = ref.float().to(torch.bfloat16).float().numpy()   # fp32 range, then bf16
    fin = np.isfinite(ref)
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    assert np.all(np.abs(y[fin] - ref[fin]) <= 2.0 ** -6 * np.abs(ref[fin]) + 1e-4)


@pytest.mark.parametrize("relu", [False, True])
def test_dense_tc_not_finite_spread(relu):
    """Several such inputs in every tile, over two filter groups and a ragged
    last tile: each output is what fp32 products and sums give."""
    g = inputs.generator(5)
    x = torch.randn(3, 3, 30, 40, generator=g)
    at = torch.rand(x.shape, generator=g)
    x[at < 0.004] = float("inf")
    x[at > 0.997] = float("-inf")
    x[(at > 0.5) & (at < 0.501)] = float("nan")
    x = x.to(torch.bfloat16)
    w = inputs.he_normal(72, 3, 7, 7, g)
    y = _run(x, w, (2, 2), (3, 3), relu)
    ref = torch.nn.functional.conv2d(x.double(), w.double(), stride=2, padding=3)
    if relu:
        ref = torch.where(ref > 0, ref, 0.0)   # NaN gives 0, as fmaxf does
    ref = ref.float().to(torch.bfloat16).float().numpy()
    fin = np.isfinite(ref)
    assert 0.1 < fin.mean() < 0.9
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    assert np.all(np.abs(y[fin] - ref[fin]) <= 2.0 ** -6 * np.abs(ref[fin]) + 1e-4)


def test_dense_tc_cost_of_not_finite_input():
    """A batch of NaN or infinities (a diverged run) costs several times a
    finite one, not hundreds: the sums end at the first NaN."""
    x = torch.randn(16, 3, 224, 224, generator=inputs.generator(6)).to(torch.bfloat16).cuda()
    w = inputs.he_normal(64, 3, 7, 7, inputs.generator(7)).cuda()
    us = []
    for xs in (x, torch.full_like(x, float("nan")), torch.full_like(x, float("inf"))):
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                y = tbn.tbn_dense_conv2d_fwd(xs, w, (2, 2), (3, 3), layout=tbn.TBN_NCHW_NHWC,
                                             out_dtype=torch.bfloat16)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 250.0)
        us.append(best)
    assert tbn.tbn_device_error() == 0
    # measured 5 and 8 times; the limit allows for other clocks and drivers
    assert max(us[1:]) <= 25.0 * us[0], us


@pytest.mark.parametrize("B,K_in,K_out", [(33, 128, 31), (1, 4, 1), (32, 129, 32), (65, 516, 100),
                                          (31, 252, 1000), (70, 1, 3), (40, 20, 33),
                                          (33, 145, 31), (9, 31, 64)])
def test_dense_linear_tile_edges(B, K_in, K_out):
    """Rows, columns and input chunks at the edges of their tiles, with
    vector (K_in % 4 == 0) and scalar loads.  fp32 sums: K_in 2^-24 sum|x w|."""
    g = inputs.generator(B * K_in)
    x = torch.randn(B, K_in, generator=g)
    w = torch.randn(K_out, K_in, generator=g)
    y = tbn.tbn_dense_linear_fwd(x.cuda(), w.cuda())
    torch.cuda.synchronize()
    want, bound = oracle.dense_linear(x.numpy(), w.numpy())
    assert np.all(np.abs(y.cpu().numpy() - want) <= K_in * 2.0 ** -24 * bound)


def test_dense_linear_pays_for_the_inputs_there_are():
    """16 inputs cost clearly less than a whole chunk of 128."""
    us = [device_us(lambda: tbn.tbn_dense_linear_fwd(x, w)) for x, w in
          ((torch.randn(10000, k, device="cuda"), torch.randn(16, k, device="cuda"))
           for k in (16, 128))]
    assert us[0] <= 0.85 * us[1], us


def test_avgpool_of_many_channels():
    """Where the threads fill the machine, more loads in flight only crowd the
    memory: four times the images, most of the first 4 us being latency, take
    less than 1.65 times as long (1.42 measured; 1.82 with 16 loads ahead)."""
    us = [device_us(lambda: tbn.tbn_avgpool2d_global_nhwc(x)) for x in
          (torch.randn(n, 7, 7, 512, device="cuda").to(torch.bfloat16) for n in (128, 512))]
    assert us[1] <= 1.65 * us[0], us


@pytest.mark.parametrize("N,H,W,C", [(3, 4, 4, 64), (2, 1, 17, 6), (5, 3, 11, 7),
                                     (128, 1, 8, 512), (33, 3, 3, 1001)])
def test_avgpool_pixel_batches(N, H, W, C):
    """Pixel counts at and off the 16 or eight loads kept in flight, odd channels."""
    x = torch.randn(N, H, W, C, generator=inputs.generator(C)).to(torch.bfloat16)
    y = tbn.tbn_avgpool2d_global_nhwc(x.cuda())
    torch.cuda.synchronize()
    want = x.double().mean((1, 2))
    tol = H * W * 2.0 ** -24 * x.double().abs().mean((1, 2)) + 2.0 ** -24 * want.abs()
    assert torch.all((y.cpu().double() - want).abs() <= tol)
