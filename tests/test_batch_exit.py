"""A CTA of the batched-decode gate/up launch does not end with a bulk copy in flight.

The copies of the LoRA-A products and RMSNorm scales complete on one mbarrier,
`aux`, which a CTA needs only when it finishes a row block.  The split of the
work leaves CTAs that finish none (their parts are added up by another CTA), so
the wait has to stand outside of every condition but that of the lane which
issued the copies.
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


def test_every_issuing_lane_waits_for_the_copies():
    text = open(SRC).read()
    issue = re.search(r"if \((NPROJ == 2 && !ROUTED && warp == LEAD && elect_one\(\))\) \{[^}]*bulk_g2s[^}]*aux\)", text)
    assert issue, "the copies' issue has changed: bring this test in line"
    tail = text[text.index("cp_async_wait_all();", issue.end()):text.index("cudaError_t launch_batch_t")]
    waits = [m.group(1).strip() for m in re.finditer(r"if \(([^;{]*?)(?: && )?!?mbar_wait\(aux, 0\)", tail)]
    assert issue.group(1) in waits, tail
