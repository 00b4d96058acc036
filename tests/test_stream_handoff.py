"""The hand-off of the stationary operand inside a CTA of the streaming kernels, as a model whose
interleavings are all explored: a wait on an mbarrier sees the parity of its completed phases only, so it
passes after one and after three phases but not after two, and a warp may look at any time or not for long.
Operands of one tile each (a head per tile) are the tightest case. The model's one parameter, who is counted
before the producer may overwrite the operand, is read from the kernel source."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_2602_02199_b200", "csrc", "stream_gemm.cuh")
N_ACC = 2              # accumulator buffers (and issuing warps)


def passes(completed, phase):
    """mbarrier parity wait for phase number `phase` when `completed` phases are over."""
    return (completed & 1) == ((phase + 1) & 1)


def stuck_states(n_tiles, issuers_counted):
    """States from which no role can move although tiles are left. Operand g serves tile g; issuing warp w
    walks every operand and multiplies the tiles of its parity. A state: operands landed, accumulators read
    out, per warp (operands looked at, tiles issued), tiles issued in order."""
    start = (0, 0, (0, 0), (0, 0))
    seen, todo, stuck = {start}, [start], []
    while todo:
        landed, drained, looked, arrived = s = todo.pop()
        nxt = []
        # producer: operand g waits for hand-back number g - 1: the epilogue has read out tile g - 1 and, if they
        # are counted, both warps have been past operand g - 1
        free = min(drained, *arrived) if issuers_counted else drained
        if landed < n_tiles and (landed == 0 or free >= landed):
            nxt.append((landed + 1, drained, looked, arrived))
        for w in range(2):
            g = looked[w]
            if g < n_tiles and arrived[w] == g and passes(landed, g):      # sees operand g
                nxt.append((landed, drained, tuple(g + 1 if i == w else x for i, x in enumerate(looked)), arrived))
            if looked[w] == arrived[w] + 1:
                t = arrived[w]                                             # its tile, if it is this warp's, and then the arrival
                if t % 2 != w or t < N_ACC or drained > t - N_ACC:
                    nxt.append((landed, drained, looked, tuple(t + 1 if i == w else x for i, x in enumerate(arrived))))
        # epilogue: tile `drained` once its warp has issued it
        if drained < n_tiles and arrived[drained % 2] > drained:
            nxt.append((landed, drained + 1, looked, arrived))
        if not nxt and min(drained, *arrived) < n_tiles:
            stuck.append(s)
        for x in nxt:
            if x not in seen:
                seen.add(x)
                todo.append(x)
    return stuck


@pytest.mark.parametrize("n_tiles", [1, 2, 3, 4, 9])
def test_no_interleaving_stalls(n_tiles):
    src = open(SOURCE).read()
    count = re.search(r"mbar_init\(bar_stat_free, ([^;]*)\);", src).group(1)
    issuers = src[src.index("MMA issuers"):src.index("epilogue warps: four groups")]
    issuers_counted = "kMmaWarps" in count and "mbar_arrive(bar_stat_free)" in issuers
    assert ("kMmaWarps" in count) == ("mbar_arrive(bar_stat_free)" in issuers)
    assert stuck_states(n_tiles, issuers_counted) == []


def test_the_model_finds_the_stall_of_uncounted_issuers():
    # the warp without a tile of operand g does not look while operands g and g + 1 land
    assert stuck_states(4, False) != []
