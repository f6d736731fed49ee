"""GPU parity of the implicit GEMM's tile shapes and epilogues against the
oracle's convolution, at the sizes where a tile, a box of filters or a
column group begins or ends.  Tolerances as in parity_util."""
import pytest
import torch

import oracle
import paper_1701_00485_gb300 as tbn
from paper_1701_00485_gb300 import inputs
from parity_util import ConvCase, assert_within

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
