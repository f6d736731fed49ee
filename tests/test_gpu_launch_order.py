"""Codes that the preceding call on the stream writes, in buffers that are
used again and again: each product equals, bit for bit, the one from codes
of their own that were complete before it was issued."""
import pytest
import torch

import paper_1701_00485_gb300 as tbn
from paper_1701_00485_gb300 import inputs

pytestmark = pytest.mark.gpu

ROUNDS = 24

CONVS = [
    # N, C, H, W, K, R, S, stride, pad
    (2, 64, 14, 14, 256, 3, 3, (1, 1), (1, 1)),     # 64-channel boxes
    (2, 96, 13, 13, 256, 3, 3, (1, 1), (1, 1)),     # 32-channel boxes
    (8, 40, 27, 27, 128, 3, 3, (1, 1), (1, 1)),     # padded channels
    (64, 64, 28, 28, 64, 3, 3, (1, 1), (1, 1)),     # row pairs
    (4, 20, 14, 14, 64, 3, 3, (3, 3), (1, 1)),      # gathered
]


def _filters(K, n, seed):
    g = inputs.generator(seed)
    return [inputs.normal((K, n), 1.2, g).cuda() for _ in range(2)]


@pytest.mark.parametrize("case", CONVS)
def test_convolution_after_its_quantizer(case):
    N, C, H, W, K, R, S, st, pd = case
    x = torch.randn(N, H, W, C, generator=inputs.generator(C)).to(torch.bfloat16).cuda()
    Ws = _filters(K, C * R * S, K + C)
    want = []
    for w in Ws:
        codes, alpha = tbn.tbn_quantize_pack(w)
        torch.cuda.synchronize()
        want.append(tbn.tbn_conv2d_fwd(x, codes, alpha, K, R, S, st, pd))
    torch.cuda.synchronize()
    got = []
    for i in range(ROUNDS):
        tbn.tbn_quantize_pack(Ws[i % 2], codes=codes, alpha=alpha)
        got.append(tbn.tbn_conv2d_fwd(x, codes, alpha, K, R, S, st, pd))
    torch.cuda.synchronize()
    assert tbn.tbn_device_error() == 0
    for i, y in enumerate(got):
        assert torch.equal(y, want[i % 2]), "round %d" % i


@pytest.mark.parametrize("case", [
    (4, 128, 16, 16, 256, 3, 3, (1, 1), (1, 1)),
    (8, 64, 20, 20, 96, 3, 3, (2, 2), (1, 1)),      # dilated dy
])
def test_input_gradients_share_a_workspace(case):
    """Two filters' transposed codes alternate in one workspace."""
    N, C, H, W, K, R, S, st, pd = case
    P, Q = tbn.conv_out_hw(H, W, R, S, st, pd)
    dy = torch.randn(N, P, Q, K, generator=inputs.generator(K)).to(torch.bfloat16).cuda()
    layers = [tbn.tbn_quantize_pack(w) for w in _filters(K, C * R * S, K + C)]
    want = []
    for codes, alpha in layers:
        want.append(tbn.tbn_conv2d_bwd_data(dy, codes, alpha, C, (H, W), R, S, st, pd))
        torch.cuda.synchronize()
    n = tbn.lib().tbn_conv2d_bwd_data_workspace_bytes(N, C, H, W, K, R, S, *st, *pd)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    got = [tbn.tbn_conv2d_bwd_data(dy, *layers[i % 2], C, (H, W), R, S, st, pd, workspace=ws)
           for i in range(ROUNDS)]
    torch.cuda.synchronize()
    assert tbn.tbn_device_error() == 0
    for i, dx in enumerate(got):
        assert torch.equal(dx, want[i % 2]), "round %d" % i


@pytest.mark.parametrize("B,K", [(1, 1024), (8, 1024), (1, 4096)])
@pytest.mark.parametrize("fp8", [False, True])
def test_linear_after_its_quantizer(B, K, fp8):
    """The GEMVs, from codes just quantized and from codes just prepared."""
    if fp8 and B > 1:
        pytest.skip("the fp8 layer takes batch 1")
    x = torch.randn(B, K, generator=inputs.generator(B)).to(torch.bfloat16).cuda()
    Ws = _filters(K, K, K)
    codes, alpha = tbn.tbn_quantize_pack(Ws[0])
    if fp8:
        prep = torch.empty(tbn.tbn_linear_f8_prepared_words(K, K), dtype=torch.int32, device="cuda")
        ws = torch.empty(tbn.tbn_linear_f8_workspace_bytes(1, K, K), dtype=torch.uint8,
                         device="cuda")

    def layer(w, wait):
        tbn.tbn_quantize_pack(w, codes=codes, alpha=alpha)
        if fp8:
            tbn.tbn_linear_prepare_f8(codes, K, out=prep)
        if wait:
            torch.cuda.synchronize()
        return (tbn.tbn_linear_fwd_f8(x, prep, alpha, K, ws) if fp8
                else tbn.tbn_linear_fwd(x, codes, alpha, K))

    want = [layer(w, True) for w in Ws]
    got = [layer(Ws[i % 2], False) for i in range(ROUNDS)]
    torch.cuda.synchronize()
    assert tbn.tbn_device_error() == 0
    for i, y in enumerate(got):
        assert torch.equal(y, want[i % 2]), "round %d" % i
