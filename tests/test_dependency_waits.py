"""Orders that no run can show to be wrong, checked in the kernels' source.

Programmatic dependent launches read nothing of the previous kernel before
griddepcontrol.wait: only behind it are that kernel's writes visible, and any
input may be one (codes come from a quantizer or from the backward pass's
transposition).  A race of this kind cannot be provoked at will, so the order
is checked in the kernels' source: in each role of a kernel that is launched
so, the wait stands before the first read of global memory."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1701_00485_gb300", "csrc")
READS = re.compile(r"__ldg\(|__ldca\(|__ldcg\(|tma_load_\w+\(|bulk_load_1d\(")

ROLES = [
    # file, where the role begins, where it ends
    ("tbn_conv_igemm.cuh", "= TMA producers =", "= gather producers ="),
    ("tbn_conv_igemm.cuh", "= gather producers =", "= patch producers ="),
    ("tbn_conv_igemm.cuh", "= patch producers =", "= MMA issuer ="),
    ("tbn_conv_igemm.cuh", "= expanders =", "= epilogue ="),
    ("tbn_conv_igemm.cuh", "= epilogue =", "- host side"),
    ("tbn_conv_smalltap.cu", "conv_smalltap_kernel(SmallTapArgs", "struct TcTile"),
    ("tbn_gemv.cu", "- producer", "- consumers"),
    ("tbn_gemv_f8.cu", "= producer: code boxes =", "} else {"),
    ("tbn_gemv_f8.cu", "// The exact three-term split of x (which", "named_barrier_sync(1, nt);"),
    ("tbn_conv_bwd.cu", "bwd_data_prep_kernel(", "struct BwdFilterArgs"),
    ("tbn_conv_bwd.cu", "bwd_filter_tma_kernel(const", "add4("),
    ("tbn_conv_bwd.cu", "bwd_filter_reduce4_kernel(\n", "bwd_filter_reduce_kernel("),
]


@pytest.mark.parametrize("name,begin,end", ROLES)
def test_wait_precedes_the_first_read(name, begin, end):
    text = open(os.path.join(CSRC, name)).read()
    assert begin in text, "role %r not found in %s" % (begin, name)
    body = text.split(begin, 1)[1]
    assert end in body, "end %r not found in %s" % (end, name)
    body = re.sub(r"//[^\n]*", "", body.split(end, 1)[0])
    wait = body.find("grid_dependency_wait();")
    first = READS.search(body)
    assert wait >= 0 and first is not None
    assert wait < first.start(), "%s: %r reads global memory before its wait" % (name, begin)


def test_rare_recomputation_is_decided_by_the_whole_warp():
    """The fp32 first layer recomputes results that are not finite and then goes
    on to warp-collective instructions (tensor-memory loads, named barriers), so
    no lane may leave the others: a vote decides, and the function that takes
    the detour ends converged."""
    text = open(os.path.join(CSRC, "tbn_dense_tc.cu")).read()
    calls = [m.start() for m in re.finditer(r"_by_taps\(", text)]
    definition, uses = calls[0], calls[1:]
    assert uses
    for u in uses:
        before = text[:u].rstrip().rsplit("\n", 2)[-2]
        assert re.search(r"if \(__any_sync\(0xffffffffu, ", before), before
    body = text[definition:text.index("\n}\n", definition)]
    assert body.rstrip().endswith("__syncwarp();")
