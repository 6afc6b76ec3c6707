"""What the roles of a GEMM kernel do to a stage's "full" barrier after a wait has expired, as a model on the CPU.

Modelled: the 512-channel pair kernel's ring (both producers, eight metadata warps, gate, MMA thread) with one stage that the
leader's producer leaves out, roles scheduled at random.  A barrier's phase stays open while its pending count or its byte
count is not zero; an arrival at a pending count of zero is beyond what the barrier was set up for and is the fault looked
for.  Whether the gate waits for the other roles to leave before it lets the MMA thread run on is read from each kernel's
source."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_15014_b200", "csrc")


class Full:
    """mbarrier with `count` arrivals per phase and a byte count that may be negative for a while."""

    def __init__(self, count):
        self.count = self.pending = count
        self.tx = self.phase = 0

    def _settle(self):
        if self.pending == 0 and self.tx == 0:
            self.phase, self.pending = self.phase + 1, self.count

    def arrive(self, expect=0):
        assert self.pending > 0, "arrival at a pending count of zero"
        self.tx += expect
        self.pending -= 1
        self._settle()

    def bytes(self, n):
        self.tx -= n
        self._settle()


def _run(seed, gate_waits, stages=6, steps=9, skipped=1, metas=8):
    rng = random.Random(seed)
    full = [Full(1 + metas) for _ in range(stages)]
    empty = [0] * stages                       # completed phases (commits)
    abort = [False]
    relay = [0]                                # steps the gate has handed over
    mma_done = [0]

    def ready(cond):                           # a role's bounded wait: success is tried before the flag is looked at
        while not cond():
            if abort[0] and rng.random() < 0.3:
                return False
            yield
        return True

    def producer(leader):
        for it in range(steps):
            s = it % stages
            if not (yield from ready(lambda: empty[s] >= it // stages)):
                return
            if leader and it == skipped:
                continue
            if leader:
                full[s].arrive(expect=2)
            yield
            full[s].bytes(1)

    def meta():
        for it in range(steps):
            s = it % stages
            if not (yield from ready(lambda: empty[s] >= it // stages)):
                return
            full[s].arrive()
            yield

    def gate():
        ok = True
        for it in range(steps):
            s, spins = it % stages, 0
            while ok and full[s].phase <= it // stages:
                spins += 1
                if spins > 400 or abort[0]:
                    abort[0], ok = True, False
                    if gate_waits:             # turns in which every other role polls, sees the flag and leaves
                        for _ in range(100):
                            yield
                yield
            if abort[0]:                       # from the expired wait on, step by step with the MMA warp
                while mma_done[0] < it:
                    yield
            relay[0] = it + 1
            yield

    def mma():
        for it in range(steps):
            while relay[0] <= it:
                yield
            yield
            empty[it % stages] += 1
            mma_done[0] = it + 1
            yield

    roles = [producer(True), producer(False), gate(), mma()] + [meta() for _ in range(metas)]
    while roles:
        r = rng.choice(roles)
        try:
            next(r)
        except StopIteration:
            roles.remove(r)
    assert abort[0]


def _gates():
    for name in ("gemm.cu", "gemm_wide.cuh", "gemm_xres.cuh"):
        src = open(os.path.join(CSRC, name)).read()
        for i, m in enumerate(re.finditer(r"-- gate\b.*?relay_step", src, re.S)):
            yield f"{name}-{i}", m.group(0)


GATES = dict(_gates())


def test_every_gemm_kernel_is_looked_at():
    assert len(GATES) == 4  # one-CTA, pair, 512-channel pair, pair with resident activations


@pytest.mark.parametrize("kernel", sorted(GATES))
def test_no_arrival_beyond_a_barriers_count_after_an_expired_wait(kernel):
    waits = re.search(r"raise_timeout\(\);\s*ptx::wait_clocks\(kGateDrain\);\s*ok = false;", GATES[kernel]) is not None
    for seed in range(200):
        _run(seed, gate_waits=waits)


def test_the_model_sees_the_fault_when_the_gate_goes_on_at_once():
    with pytest.raises(AssertionError, match="pending count of zero"):
        for seed in range(200):
            _run(seed, gate_waits=False)


def _run_split(seed, kblocks=9, stages=4, skipped=1, ctas=3, builders=4, tells=True):
    """The split kernel: CTA 0's producer leaves one stage out.  No gate: the MMA thread waits itself and stops for good, its epilogue warps
    then fail.  Returns, per CTA, whether it writes outputs, and which CTAs' sums it has."""
    rng = random.Random(seed)
    full = [[Full(1 + builders) for _ in range(stages)] for _ in range(ctas)]
    empty = [[0] * stages for _ in range(ctas)]
    abort, acc, failed = [False] * ctas, [False] * ctas, [False] * ctas
    met, sums, wrote = [0, 0], [set() for _ in range(ctas)], [None] * ctas

    def ready(c, cond, patience=4000):
        spins = 0
        while not cond():
            spins += 1
            if (abort[c] and rng.random() < 0.3) or spins > patience:
                return False
            yield
        return True

    def producer(c, expects):  # of X, with bytes to come, or a builder warp
        for it in range(kblocks):
            s = it % stages
            if not (yield from ready(c, lambda: empty[c][s] >= it // stages)):
                abort[c] = True
                return
            if c == 0 and it == skipped and expects:
                continue
            full[c][s].arrive(expect=1 if expects else 0)
            yield
            if expects:
                full[c][s].bytes(1)

    def mma(c):
        for it in range(kblocks):
            if not (yield from ready(c, lambda: full[c][it % stages].phase > it // stages, 600)):
                abort[c] = True
                return
            empty[c][it % stages] += 1
            yield
        acc[c] = True

    def epilogue(c):
        ok = yield from ready(c, lambda: acc[c])
        abort[c] = abort[c] or not ok
        for step in range(2):
            met[step] += 1
            while met[step] < ctas:           # the cluster's barriers: everyone arrives, flag or not
                yield
            if step == 0:
                for r in range(ctas):
                    if ok:
                        sums[r].add(c)
                    elif tells:
                        abort[r] = True
                yield
        wrote[c] = ok and not abort[c]

    roles = [g for c in range(ctas) for g in [producer(c, True), mma(c), epilogue(c)] + [producer(c, False) for _ in range(builders)]]
    while roles:
        r = rng.choice(roles)
        try:
            next(r)
        except StopIteration:
            roles.remove(r)
    return wrote, sums


def test_split_kernel_writes_nothing_once_a_cta_has_given_up():
    src = open(os.path.join(CSRC, "gemm_split.cuh")).read()
    exchange = src[src.index("ptx::cluster_wait();"):src.index("const float rsy")]  # from the first cluster barrier to the outputs
    send, finish = exchange.split("ptx::cluster_arrive();")
    tells = "st_cluster_u32(ptx::map_to_cta(ptx::smem_u32((const void*)abort_flag)" in send and "const bool whole = *abort_flag == 0u;" in finish and "jmax = whole &&" in src
    for seed in range(30):
        wrote, sums = _run_split(seed, tells=tells)
        assert not any(w and len(s) < len(sums) for w, s in zip(wrote, sums)), "outputs from sums that were never sent"
    assert any(any(_run_split(seed, tells=False)[0]) for seed in range(30))  # the model sees the fault
    wrote, sums = _run_split(1, skipped=-1)
    assert all(wrote) and all(len(s) == 3 for s in sums)
