"""The order of work of the 64-dimensional SM-pair kernel, followed on the CPU.

A wait by parity tells a barrier's last completed phase from the one before it
only, so no barrier may complete twice before all its waiters have seen the
first time: a late waiter would then wait for a phase that needs the waiter
itself.  The MMA warp issues its items in order and knows of the epilogue warps
only what its own waits imply; here they are as late as these waits allow, and
the barrier of every score commit comes from the kernel's own text."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_07144_gb300", "csrc")


def _kernel():
    text = open(os.path.join(CSRC, "rvq.cu")).read()
    text = text[text.index("k_rvq64_pair("):]
    return text[:text.index("\n}\n")]


def _acc_barrier(text, call):
    """The one expression whose barrier `call` names, as a function of (k, blk)."""
    exprs = set(re.findall(re.escape(call) + r"\(bar\(BAR_ACC \+ ((?:[^()]|\([^()]*\))*)\)", text))
    assert len(exprs) == 1, exprs
    code = compile(exprs.pop(), "rvq.cu", "eval")
    return lambda k, blk: eval(code, {"k": k, "blk": blk})


@pytest.mark.parametrize("blocks", [1, 4])
def test_no_score_barrier_runs_ahead_of_its_waiters(blocks):
    text = _kernel()
    commit, wait = _acc_barrier(text, "umma_commit_pair"), _acc_barrier(text, "wait_or_abort")
    free = "(n < 2 || wait_or_abort(bar(BAR_FREE + (n & 1)), ((n >> 1) - 1) & 1,"
    ready = "if (blk == 0) {\n                                ok = wait_cluster(bar(BAR_READY + k)"
    assert free in text and ready in text         # the two waits followed below
    slots = 3
    for stages in (1, 2, 4):
        for units in range(1, 8):
            n = 0
            items = []                            # slot of item n
            seen = [0] * slots                    # the slot's items that its warps are known to have read
            issued = [0] * slots
            pending = {}                          # barrier -> the slot's item count at its last commit
            for first in range(0, units, slots):
                act = min(slots, units - first)
                for s in range(stages):
                    for blk in range(blocks):
                        for k in range(act):
                            if blk == 0:          # a_ready: all the slot's scores before are read
                                seen[k] = issued[k]
                            if n >= 2:            # acc_free: so are item n - 2's, and its slot's before them
                                j, count = items[n - 2]
                                seen[j] = max(seen[j], count)
                            issued[k] += 1
                            items.append((k, issued[k]))
                            bar = commit(k, blk)
                            assert bar == wait(k, blk)
                            assert pending.get(bar, (k, 0))[0] == k, "a barrier of two slots"
                            assert pending.get(bar, (k, 0))[1] <= seen[k], (stages, units, n)
                            pending[bar] = (k, issued[k])
                            n += 1
