"""The exact path's tensor-core kernel hands kernel boxes to two groups of warps in turn through a ring of slots.  A model of the ring on
the CPU: barriers as phase counters that answer a parity wait as the hardware does (true when the current phase's parity differs), boxes
that land in any order, groups that run as far ahead as their other waits let them.  A group must never take a box that is not there."""
import itertools
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1611_07151_b200", "csrc", "conv_f32_tc.cu")


def run(slots, units, order, guarded):
    """Boxes land in `order`; between two landings both groups and the producer go on as far as they can.  True: no wrong box was taken."""
    landed_phase = [0] * slots              # completed phases of full[s]
    given_back = [0] * slots                # completed phases of empty[s]
    issued, taken, mma_done = 0, [0, 1], -1     # next box to issue, next unit per group, last unit whose MMAs are done
    stored = set()                          # units whose split kernels are in TMEM
    holds = [False, False]                  # a group has read its unit's box and waits for the kernel slot in TMEM
    pending = []
    passed = lambda phases, parity: (phases & 1) != parity      # mbarrier.try_wait.parity
    landings = iter(order)
    while True:
        moved = True
        while moved:
            moved = False
            if issued < units and (issued < slots or given_back[issued % slots] >= issued // slots):
                pending.append(issued)
                issued += 1
                moved = True
            for g in (0, 1):
                u = taken[g]
                if holds[g]:
                    if mma_done >= u - 2:
                        stored.add(u)
                        holds[g], taken[g] = False, u + 2
                        moved = True
                    continue
                if u >= units:
                    continue
                s, k = u % slots, u // slots
                if guarded and slots % 2 and mma_done < u - slots:
                    continue
                if not passed(landed_phase[s], k & 1):
                    continue
                if landed_phase[s] != k + 1:
                    return False                        # not this unit's box
                given_back[s] += 1
                holds[g] = moved = True
            while mma_done + 1 in stored:
                mma_done += 1
                moved = True
        if not pending:
            return taken[0] >= units and taken[1] >= units
        first = next((b for b in landings if b in pending), None)
        b = first if first is not None else pending[0]
        pending.remove(b)
        landed_phase[b % slots] += 1


@pytest.mark.parametrize("slots", [2, 3, 4])
def test_no_box_is_taken_early(slots):
    units = 7
    for order in itertools.permutations(range(units)):
        assert run(slots, units, order, guarded=True), order


def test_the_model_sees_what_an_odd_ring_does_without_the_guard():
    """Three slots, unit 2's box before unit 1's: unit 4 takes slot 1 while it is empty."""
    assert not run(3, 7, (0, 2, 1, 3, 4, 5, 6), guarded=False)


def test_the_kernel_is_the_one_that_is_modelled():
    """The slot counts of the kernel's rings are those above, and its guard stands before the wait for the box."""
    text = open(SOURCE).read()
    boxes = {int(n) for name in ("flat", "patch", "box") for n in re.findall(r"{\d, \d, (\d)}", re.search(r"\b%s\[\]\[3\] = {(.*?)}[,;]" % name, text).group(1) + "}")}
    assert boxes and boxes <= {2, 3, 4}, boxes
    guard = text.index("if ((p.sb & 1) && !wait_done(u - p.sb)) break;")
    wait = text.index("wait_bar(smem_u32(&sh->sb_full[st]), sph")
    assert 0 < wait - guard < 200 and text.count("sb_full[st]), sph") == 1
