"""The named barriers of a block in the decoder kernel, on the CPU.  A hardware barrier counts arrivals and does not
know whose they are: a warp that arrives twice stands in for one that has not come yet.  Here the 16 warps of
a CTA take the steps of a block around the QKV GEMM in every order of a slow and a fast warp, with the barrier
numbers that the kernel's source has."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2410_05911_gb300", "csrc", "decoder_kernel.cuh")
WARPS = 16


def barrier_numbers():
    """(the barrier that warp 0 arrives at when the accumulators are complete, where the others wait for it, the
    CTA-wide barrier after the K/V epilogue)"""
    with open(SRC) as f:
        s = f.read()
    consts = dict(re.findall(r"constexpr uint32_t (k\w+Bar) = (\d+);", s))
    number = lambda name: int(consts.get(name, name))  # noqa: E731
    arrive = {number(x) for x in re.findall(r"release_acc\(\) \{ named_bar_arrive\((\w+), kEpiThreads\)", s)}
    wait = {number(x) for x in re.findall(r"if \(warp != 0\) named_bar_sync\((\w+), kEpiThreads\)", s)}
    cta = {number(x) for x in re.findall(r"named_bar_sync\((\w+), kEpiThreads\);  // every Q, K, V row", s)}
    assert len(arrive) == len(wait) == len(cta) == 1
    return arrive.pop(), wait.pop(), cta.pop()


class Bar:
    def __init__(self):
        self.count, self.phase = 0, 0

    def arrive(self):
        """One warp's arrival; the phase that it belongs to."""
        phase = self.phase
        self.count += 1
        if self.count == WARPS:
            self.count, self.phase = 0, self.phase + 1
        return phase


def run(order, blocks=3):
    """Let the warps advance in the given order of preference until all have finished `blocks` blocks or none can;
    returns whether they finished and whether a warp ever left the K/V barrier before every warp had come."""
    acc_arrive, acc_wait, cta = barrier_numbers()
    bars = {b: Bar() for b in (acc_arrive, acc_wait, cta)}
    published = 0           # operands published over all warps (an mbarrier: 16 a block)
    steps = ("publish", "accumulators", "keys and values", "attention")
    at = [0] * WARPS        # step counter of each warp
    held = [None] * WARPS   # (barrier, phase) that the warp waits in
    came = [0] * (blocks * 2)
    early = False
    while True:
        for w in order:
            if held[w] is not None and bars[held[w][0]].phase > held[w][1]:
                b, name, blk = held[w][0], steps[at[w] % 4], at[w] // 4
                if name in ("keys and values", "attention"):
                    early |= came[2 * blk + (name == "attention")] < WARPS
                held[w] = None
                at[w] += 1
                break
            if held[w] is not None or at[w] == 4 * blocks:
                continue
            name, blk = steps[at[w] % 4], at[w] // 4
            if name == "publish":
                published += 1
                at[w] += 1
                break
            if name == "accumulators":
                if w == 0:
                    if published < WARPS * (blk + 1):
                        continue  # warp 0 issues the GEMM once every warp has published its part
                    bars[acc_arrive].arrive()
                    at[w] += 1
                else:
                    held[w] = (acc_wait, bars[acc_wait].arrive())
                break
            came[2 * blk + (name == "attention")] += 1
            held[w] = (cta, bars[cta].arrive())
            break
        else:
            return all(a == 4 * blocks for a in at), early


@pytest.mark.parametrize("fast", [0, 1, 15])
@pytest.mark.parametrize("slow", [1, 7, 15])
def test_no_arrival_stands_in_for_a_late_warp(fast, slow):
    if fast == slow:
        pytest.skip("one warp")
    order = [fast] + [w for w in range(WARPS) if w not in (fast, slow)] + [slow]
    done, early = run(order)
    assert done and not early
