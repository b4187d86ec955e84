"""Model check of the bounded waits of the fixed-point march with per-step factors.

A system of W warps in one CTA marches nt steps.  Each step every warp waits for the step's rows
(a bulk copy that the first warp asked for a step earlier), meets the others at a barrier and goes
on; the first warp then asks for the next step's rows.  A wait that runs out must end the march of
the whole system: the barrier itself has no limit, so no warp may leave while another goes on to
it.  The copy of one step arrives late or never, and each warp's wait gives up, or is served, in
any order.

The model runs the kernel's rule (the warps' give-up flags are combined by the barrier, and all
leave behind it) under random schedules, and shows that the rule it replaced (a warp whose wait
runs out leaves its loop at once) can leave warps at the barrier for ever.  It models the design,
not the CUDA code, and needs no GPU."""
import random

import pytest


class Hang(AssertionError):
    pass


def _run(W, nt, late_step, arrives, rng, leave_at_once=False):
    """One random schedule; the step each warp left after (nt: it finished)."""
    step, phase = [2] * W, ["wait"] * W
    gave_up = [False] * W
    left = [None] * W
    there = {2} if late_step != 2 else set()
    asked = {2}
    while any(x is None for x in left):
        moves = []
        for w in range(W):
            if left[w] is not None:
                continue
            t = step[w]
            if phase[w] == "wait":
                if t in there:
                    moves.append((w, "served"))
                elif t == late_step:
                    moves.append((w, "out"))      # the limit
        at = [w for w in range(W) if left[w] is None and phase[w] == "bar"]
        if len(at) == W:                          # the barrier wants every warp of the system
            moves.append((-1, "release"))
        if late_step in asked and late_step not in there and arrives:
            moves.append((-1, "arrive"))
        if not moves:
            raise Hang(f"steps {step}, phases {phase}, left {left}")
        w, what = rng.choice(moves)
        if what == "arrive":
            there.add(late_step)
        elif what == "served":
            phase[w] = "bar"
        elif what == "out":
            gave_up[w] = True
            if leave_at_once:
                left[w] = step[w]
            else:
                phase[w] = "bar"
        else:
            any_late = any(gave_up)               # the barrier's reduction
            t = step[0]
            assert len(set(step)) == 1
            for k in range(W):
                if any_late or t == nt:
                    left[k] = t
                else:
                    step[k], phase[k] = t + 1, "wait"
            if not any_late and t < nt:
                asked.add(t + 1)
                if t + 1 != late_step:
                    there.add(t + 1)
    return left, gave_up


@pytest.mark.parametrize("W", [2, 3, 6, 12])
@pytest.mark.parametrize("arrives", [True, False])
def test_all_warps_leave_together(W, arrives):
    rng = random.Random(W)
    for _ in range(200):
        nt = rng.randint(2, 9)
        late = rng.randint(2, nt)
        left, gave_up = _run(W, nt, late, arrives, rng)
        assert len(set(left)) == 1
        if any(gave_up):
            assert left[0] == late
        else:
            assert left[0] == nt


def test_leaving_at_once_can_hang():
    rng = random.Random(3)
    hangs = 0
    for _ in range(200):
        try:
            _run(4, 6, 4, True, rng, leave_at_once=True)
        except Hang:
            hangs += 1
    assert hangs
