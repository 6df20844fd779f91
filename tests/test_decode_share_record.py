"""The decoder CTA's record of its share of a step (shared memory, kShares
copies): every order in which the warps of a CTA can reach their accesses.

A warp writes the next step's share while it schedules (the last warp only
arrives at the grid barrier), meets the others at the barrier that ends the
step, and reads its share behind it.  A CTA whose share is empty meets no other
barrier in between.  The model runs those accesses for every interleaving and
every pattern of empty shares and checks that each warp reads its own step's
share; the number of copies is the source's.
"""
import itertools
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2201_05213_gb300", "csrc",
                   "nlc_decode_kernel.cuh")


def copies():
    text = open(SRC).read()
    m = re.search(r"constexpr int kShares = (\d+);", text)
    assert m and "[(unsigned)step % kShares]" in text
    return int(m.group(1))


def program(pixels, schedules):
    """One warp's accesses: write / read of a step's share, 'bar' a CTA barrier."""
    ops = [("write", 0), ("bar",), ("read", 0)]
    for step, n in enumerate(pixels):
        if n:
            ops.append(("bar",))  # the barriers inside a tile
        if step + 1 < len(pixels):
            if schedules:
                ops.append(("write", step + 1))
            ops += [("bar",), ("read", step + 1)]
    return ops


def wrong_reads(pixels, n_copies):
    """Reads of another step's share over all interleavings of three warps."""
    progs = [program(pixels, True), program(pixels, True), program(pixels, False)]
    start = ((0, 0, 0), (None,) * n_copies)
    seen, todo, wrong = {start}, [start], set()
    while todo:
        pcs, mem = todo.pop()
        nexts = []
        at = [progs[w][pc] if pc < len(progs[w]) else None for w, pc in enumerate(pcs)]
        if all(a == ("bar",) for a in at):
            nexts.append((tuple(pc + 1 for pc in pcs), mem))
        for w, a in enumerate(at):
            if a is None or a == ("bar",):
                continue
            m = mem
            if a[0] == "write":
                m = tuple(a[1] if i == a[1] % n_copies else v for i, v in enumerate(mem))
            elif mem[a[1] % n_copies] != a[1]:
                wrong.add((a[1], mem[a[1] % n_copies]))
            nexts.append((tuple(pc + (i == w) for i, pc in enumerate(pcs)), m))
        for s in nexts:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return wrong


@pytest.mark.parametrize("pixels", list(itertools.product((0, 1), repeat=5)))
def test_every_warp_reads_its_own_steps_share(pixels):
    assert not wrong_reads(pixels, copies())


def test_the_model_finds_the_hazard_of_a_single_copy():
    assert wrong_reads((0, 1, 1), 1)
    assert not wrong_reads((1, 1, 1), 1)  # only an empty share lacks the barrier
