"""A bounded wait may run out on some lanes of a warp and not on others.  Where a whole warp
waits and then runs warp-wide instructions (reads of tensor memory, full-mask shuffles), the
lanes agree on the outcome first, so that they leave or go on together."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_00548_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_drain_warps_of_the_slice_product_agree():
    drain = _code("residual_oz.cu").split("const int quarter")[1].split("bool drained")[0]
    waits = re.findall(r"[^\n;{}]*mbar_wait\([^\n]*", drain)
    assert len(waits) == 1 and "__all_sync(0xffffffffu, mbar_wait(" in waits[0]
    assert drain.index("mbar_wait(") < drain.index("tmem_ld16(") < drain.index("__shfl_sync(")


def test_block_agrees_in_the_tensor_core_product():
    body = _code("cgemm_tc.cu").split("k_cgemm_tc(const CGemmArgs G")[1]
    assert re.search(r"ok = mbar_wait\([^\n]*\n\s*ok = __syncthreads_and\(ok\)", body)
