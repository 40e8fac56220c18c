"""The waits between the warps of the GPTQ kernel (csrc/gptq.cu), as a model: updating warps hand a block over through one barrier, `ready`, rounding
warps a group of it through another each, `done`, and a wait knows a phase by its parity alone.  Every order in which the warps can get on is
walked through: none ends with a warp that waits for good, and no wait passes on another phase's account.  The first block may have fewer groups
than there are rounding warps."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_14363_b200", "csrc", "gptq.cu")


def _programs(updating, rounding, groups, first, blocks, seen):
    """A list of steps per warp: ("wait", barrier, parity, phase) or ("arrive", barrier).  `seen`: a rounding warp without a group in the first block
    arrives on `ready` at its start and whenever it has seen a phase of it."""
    count = lambda b: first if b == 0 else groups
    phase = lambda g, b: b - (1 if g >= first else 0)  # of group g in block b; groups beyond the first block's start a block later
    parity = lambda g, b: (b + (1 if g >= first else 0)) & 1  # done_parity
    done = lambda g, b: ("wait", 1 + g, parity(g, b), phase(g, b))
    programs = []
    for _ in range(updating):
        programs.append([step for b in range(blocks) for step in [done(g, b - 1) for g in range(count(b - 1) if b else 0)] + [("arrive", 0)]])
    for w in range(rounding):
        says = [("arrive", 0)] if seen and w >= first else []
        steps = list(says)
        for b in range(blocks):
            steps += [("wait", 0, b & 1, b)] + says
            for g in range(w, count(b), rounding):
                steps += [done(before, b) for before in range(g)] + [("arrive", 1 + g)]
        programs.append(steps)
    return programs


def _closed(updating, rounding, groups, first, blocks, seen):
    programs = _programs(updating, rounding, groups, first, blocks, seen)
    needs = [updating + (max(rounding - first, 0) if seen else 0)] + [1] * groups
    start = ((0,) * len(programs), ((0, 0),) * (1 + groups))  # places in the programs; (phases completed, arrivals of the next) per barrier
    todo, known = [start], {start}
    while todo:
        at, bars = todo.pop()
        moved = False
        for w, program in enumerate(programs):
            if at[w] == len(program):
                continue
            kind, bar, *rest = program[at[w]]
            completed, arrived = bars[bar]
            if kind == "wait":
                if (completed & 1) == rest[0]:  # a parity is passed while the phase under way has the other one
                    continue
                if completed != rest[1] + 1:
                    return False  # passed on another phase's account
                new = bars
            else:
                state = (completed + 1, 0) if arrived + 1 == needs[bar] else (completed, arrived + 1)
                new = bars[:bar] + (state,) + bars[bar + 1:]
            moved = True
            nxt = (at[:w] + (at[w] + 1,) + at[w + 1:], new)
            if nxt not in known:
                known.add(nxt)
                todo.append(nxt)
        if not moved and any(a < len(p) for a, p in zip(at, programs)):
            return False
    return True


@pytest.mark.parametrize("first", [1, 2, 3, 4])
def test_every_order_of_the_warps_ends(first):
    assert _closed(1, 2, 4, first, 4, seen=True)
    assert _closed(2, 2, 4, first, 3, seen=True)
    assert _closed(1, 3, 3, min(first, 3), 3, seen=True)


def test_a_warp_that_only_looks_on_can_miss_a_phase():
    assert _closed(1, 2, 4, 2, 3, seen=False)  # a group for every warp
    assert not _closed(1, 2, 4, 1, 3, seen=False)


def test_the_kernel_waits_as_the_model_does():
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    assert "mbar_init(&ready, kWarps + max(kWarps - first_groups, 0));" in text and "mbar_init(&done[g], 1);" in text
    updating, rounding = text.split("if (warp < kWarps) {", 1)[1].split("} else {", 1)
    assert updating.count("mbar_arrive(&ready)") == 1
    # a rounding warp: at its start, and behind the one place where it waits
    assert "const bool onlooker = warp - kWarps >= first_groups;" in rounding
    assert rounding.count("if (onlooker && lane == 0) mbar_arrive(&ready);") == rounding.count("mbar_arrive(&ready)") == 2
    assert rounding.count("warp_wait(&ready") == 1 and "done_parity(before, b)" in rounding
    assert re.search(r"if \(!warp_wait\(&ready, b & 1\)\) return false;\s*if \(onlooker && lane == 0\) mbar_arrive\(&ready\);\s*return true;", rounding)
    assert len(re.findall(r"!block_ready\(b\)\) goto failed;", rounding)) == 2
    assert "return static_cast<uint32_t>(b + (g >= first_groups ? 1 : 0)) & 1u;" in text
