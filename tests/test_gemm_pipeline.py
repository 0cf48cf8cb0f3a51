"""The hand-overs of the stream-K prefill GEMM (qgemm_sk_kernel), as a model on the CPU.

A CTA computes the parts of tiles in its range one after another into the same
accumulators.  Two groups of dequantizing warps make alternate stages of a part;
every warp reads its share of the finished accumulators.  Nothing but the waits
orders the next part's first MMA after those reads, so the model runs the roles
in random order and at random speeds and checks that no warp reads sums of
another part.  What the MMA role waits for is taken from the kernel's source.
"""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_04238_gb300", "csrc",
                   "wq_gemm.cu")
WARPS, GROUP = 16, 8


class Barrier:
    """An mbarrier: completed phases, and the arrivals missing in the present one."""

    def __init__(self, count):
        self.count = self.missing = count
        self.phase = 0

    def arrive(self):
        self.missing -= 1
        if self.missing == 0:
            self.phase, self.missing = self.phase + 1, self.count

    def done(self, parity):
        return (self.phase & 1) != parity


def run(parts, slots, wait_empty, seed):
    """`parts`: stages of each part.  Raises AssertionError when a warp reads another part's sums."""
    rnd = random.Random(seed)
    b_full = [Barrier(GROUP) for _ in range(slots)]
    b_empty = [[Barrier(1), Barrier(1)] for _ in range(slots)]  # even and odd uses
    acc_full, acc_empty = Barrier(1), Barrier(WARPS)
    acc = dict(part=-1, stages=0)
    queue = []  # issued MMAs and commits, in order

    def mma():
        st = 0
        for part, nit in enumerate(parts):
            while wait_empty and part > 0 and not acc_empty.done((part - 1) & 1):
                yield
            for it in range(nit):
                while not b_full[st % slots].done((st // slots) & 1):
                    yield
                queue.append((part, it, st))
                st += 1
                yield
            queue.append((part, None, None))

    def tensor_pipe():
        while True:
            if queue:
                part, it, st = queue.pop(0)
                if it is None:
                    acc_full.arrive()
                else:
                    acc.update(part=part, stages=it + 1)
                    b_empty[st % slots][(st // slots) & 1].arrive()
            yield

    def warp(w):
        base = 0
        for part, nit in enumerate(parts):
            for it in range(w // GROUP, nit, 2):
                st = base + it
                use = st // slots - 1
                while use >= 0 and not b_empty[st % slots][use & 1].done((use >> 1) & 1):
                    yield
                yield
                b_full[st % slots].arrive()
            base += nit
            while not acc_full.done(part & 1):
                yield
            for _ in range(4):  # the reads of this warp's columns
                assert acc == dict(part=part, stages=nit), "sums of another part read"
                yield
            acc_empty.arrive()

    roles = [mma(), tensor_pipe()] + [warp(w) for w in range(WARPS)]
    # the second group's warps up to 8 times slower
    speed = [1.0, 1.0] + [rnd.uniform(0.3, 1.0) / (rnd.uniform(1, 8) if w >= GROUP else 1) for w in range(WARPS)]
    alive = [0] + list(range(2, 2 + WARPS))
    for _ in range(200000):
        if not alive:
            return
        live = alive + [1]
        i = rnd.choices(live, [speed[j] for j in live])[0]
        try:
            next(roles[i])
        except StopIteration:
            alive.remove(i)
    raise AssertionError("a wait that never ends")


def schedules():
    for seed in range(150):
        rnd = random.Random(1000 + seed)
        yield [rnd.choice([1, 2, 3, 4, 8]) for _ in range(rnd.randint(2, 4))], rnd.choice([2, 3]), seed


def source_waits_for_reads():
    """Whether the MMA role waits for the 16 warps' reads before a later part's first MMA."""
    text = open(SRC).read()
    body = text[text.index("qgemm_sk_kernel("):text.index("#undef WQ_FOR_EACH_PART")]
    role = body[body.index("warp == kMmaWarp"):]
    before = role[:role.index("gemm_issue_stage")]
    init = re.search(r"mbar_init\(acc_empty,\s*kDeqWarps\)", text)
    arrive = role.find("mbar_arrive(sm.acc_empty)") > role.find("gemm_part_epilogue")
    return bool(init) and "wait(sm.acc_empty, (part - 1) & 1)" in before and arrive


def test_parts_do_not_overwrite_sums_that_are_still_read():
    wait = source_waits_for_reads()
    for parts, slots, seed in schedules():
        run(parts, slots, wait, seed)


def test_the_model_sees_the_missing_wait():
    def fails(parts, slots, seed):
        try:
            run(parts, slots, False, seed)
        except AssertionError:
            return True
        return False
    assert sum(fails(*s) for s in schedules()) > 20
    with pytest.raises(AssertionError, match="another part"):
        for parts, slots, seed in schedules():
            run(parts, slots, False, seed)


def test_a_timeout_settles_before_the_cta_ends():
    """Both kernels: a CTA that met a timeout gives the loads and MMAs of its other roles
    time to end before it frees its tensor memory and leaves."""
    text = open(SRC).read()
    ends = re.findall(r"  if \(\*sm\.abort_s\) gemm_settle\(\);\n  tc_fence_before\(\);\n  __syncthreads\(\);\n  tc_fence_after\(\);"
                      r"\n  if \(warp == kMmaWarp\) tmem_dealloc\(tmem", text)
    assert len(ends) == 2 and text.count("tmem_dealloc(tmem") == 2
