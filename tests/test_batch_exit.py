"""A CTA of the batched-decode gate/up launch does not end with a bulk copy in flight.

The copies of the LoRA-A products and RMSNorm scales complete on one mbarrier,
`aux`, which a CTA needs only when it finishes a row block.  The split of the
work leaves CTAs that finish none (their parts are added up by another CTA), so
a wait at the end of the CTA has to stand outside of every condition.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_04238_gb300", "csrc",
                   "wq_batch.cuh")


def may_finish_nothing(n, k, sms):
    """CTAs whose row blocks are all split: whichever of a block's CTAs comes last finishes it."""
    u, t = (k + 127) // 128, (n + 127) // 128
    w = t * u
    p = max(1, min(sms, w // 2))
    out = 0
    for c in range(p):
        g0, g1 = w * c // p, w * (c + 1) // p
        out += not any(g0 <= b * u and (b + 1) * u <= g1 for b in range(g0 // u, (g1 - 1) // u + 1))
    return out


@pytest.mark.parametrize("n,k", [(14336, 4096), (9728, 2560), (10624, 704)])
def test_some_ctas_may_finish_no_row_block(n, k):
    assert may_finish_nothing(n, k, 152) > 0


def test_thread_0_waits_for_the_copies():
    """A CTA's shared memory stays its own until all of its threads are done, so one
    thread's wait suffices."""
    text = open(SRC).read()
    assert text.count("bulk_g2s(smem + C::OFF_TF, a.tfrag, tfb, aux)") == 1, "the copies' issue has changed"
    kernel = text[text.index("batch_kernel(const __grid_constant__ BatchArgs a)"):text.index("cudaError_t launch_batch_t")]
    tail = kernel[kernel.rindex("cp_async_wait_all();"):]
    assert re.search(r"\n  if \(NPROJ == 2 && !ROUTED && tid == 0 && !mbar_wait\(aux, 0\)\)", tail), tail
    # nothing returns before it
    assert not re.search(r"\n\s*(?:if \([^;]*\) )?return;", kernel[kernel.index("mbar_arrive_expect_tx(aux"):])
