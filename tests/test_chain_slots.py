"""The block slots of the chain kernel's last streamer, as a model on the CPU: its loader, sender and
group and the CTA that the blocks go on to, in every order that the waits allow.  Waits are by parity, as
on the GPU: one that comes two phases late looks like one that comes too early."""
import os
import re

import pytest

STREAM = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_22099_gb300", "csrc",
                      "gbtrf_wide_stream.cuh")


def first_stuck_state(streamers, slots, blocks, free_arrivals):
    """Explores every interleaving.  None when all agents always finish with every wait passed in its own
    phase, else what went wrong first.  A block b < streamers has no panel here: the sender alone moves it."""
    names = ("loader", "sender", "group", "credit")
    start = (1,) * len(names) + (0,)  # the agents' next blocks; 1 while the group is past its first wait

    def phases(state, kind, slot):
        # phases completed on the slot's barrier: one for each of the slot's blocks that an agent is through
        def done(agent_next):
            return sum(1 for b in range(1, agent_next) if (b - 1) % slots == slot)
        loader, sender, group, credit, _ = state
        if kind == "in":
            return done(loader)
        if kind == "dst":
            return done(sender)
        return done(credit) if free_arrivals == 1 else min(done(credit), done(group))

    def passes(state, kind, b):
        """Whether a wait for block b's event passes, and whether that is its own phase."""
        event, c = (b - 1) // slots, phases(state, kind, (b - 1) % slots)
        return (c - event) % 2 == 1, c == event + 1

    seen, todo = {start}, [start]
    while todo:
        state = todo.pop()
        loader, sender, group, credit, half = state
        steps = []
        if loader <= blocks:
            if loader <= slots:
                steps.append(((loader + 1, sender, group, credit, half), True))
            else:
                go, own = passes(state, "free", loader - slots)
                if go:
                    steps.append(((loader + 1, sender, group, credit, half), own))
        if sender <= blocks:
            go, own = passes(state, "in", sender)
            if go:
                steps.append(((loader, sender + 1, group, credit, half), own))
        if group <= blocks:
            go, own = passes(state, "dst" if half else "in", group)
            if go:
                steps.append(((loader, sender, group + half, credit, 1 - half), own))
        if credit < sender and (credit < streamers or credit < group):
            steps.append(((loader, sender, group, credit + 1, half), True))
        if not steps and min(loader, sender, group, credit) <= blocks:
            return f"stuck at {dict(zip(names, state))}"
        for nxt, own in steps:
            if not own:
                return f"a wait passed in the wrong phase at {dict(zip(names, state))}"
            if nxt not in seen:
                seen.add(nxt)
                todo.append(nxt)
    return None


def free_arrivals_of_the_kernel():
    with open(STREAM) as f:
        return int(re.search(r"kFreeArrivals = (\d+);", f.read()).group(1))


@pytest.mark.parametrize("streamers,slots", [(7, 4), (5, 3), (4, 3)])
def test_the_last_streamers_group_misses_no_block(streamers, slots):
    assert first_stuck_state(streamers, slots, 20, free_arrivals_of_the_kernel()) is None
    # freed by the credit alone, a slot could be filled twice before the group looked at it
    assert "stuck" in first_stuck_state(streamers, slots, 20, 1)
