"""The barriers through which the store warp learns that an item has been stored, where the epilogue stores by itself: every order
in which scheduler, epilogue and store warp can take their steps, with the ring lengths of the kernel source.

The store warp hands the ring slot of item n back when it takes the item and only then waits for the item's barrier, so the others
can run ahead of it.  A barrier that has completed twice by the time the store warp looks has the parity it had before: the wait
would run into its time-out."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_26842_b200", "csrc", "ns_tc.cu")


def reaches_a_missed_phase(ring, done_ring, items):
    """Whether some order of steps lets item n's barrier complete a second time while the store warp is still to see the first.
    A state: items published, items taken and items stored by the epilogue, items taken and items seen stored by the store warp."""
    seen, todo = set(), [(0, 0, 0, 0, 0)]
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        published, taken, stored, store_taken, store_seen = state
        if published < items and published - min(taken, store_taken) < ring:      # the slot has been handed back by both readers
            todo.append((published + 1, taken, stored, store_taken, store_seen))
        if taken < published and taken == stored:
            todo.append((published, taken + 1, stored, store_taken, store_seen))
        if stored < taken:
            todo.append((published, taken, stored + 1, store_taken, store_seen))
        if store_taken == store_seen:
            if store_taken < published:
                todo.append((published, taken, stored, store_taken + 1, store_seen))
            continue
        n = store_seen                                                            # the item the store warp is waiting for
        completions = len(range(n % done_ring, stored, done_ring))
        if completions >= n // done_ring + 2:
            return True
        if completions == n // done_ring + 1:
            todo.append((published, taken, stored, store_taken, store_seen + 1))
    return False


def constant(name, known={}):
    value = re.search(rf"constexpr int {name} = ([^;]+);", open(SOURCE).read()).group(1)
    return eval(value, {}, known)


def test_no_order_of_steps_lets_the_store_warp_miss_an_item():
    ring = constant("RING")
    done_ring = constant("DONE_RING", {"RING": ring})
    assert not reaches_a_missed_phase(ring, done_ring, 4 * done_ring)


@pytest.mark.parametrize("ring,done_ring,missed", [(4, 4, True), (4, 5, False), (2, 2, True), (2, 3, False), (1, 1, True)])
def test_the_model_tells_safe_lengths_from_unsafe_ones(ring, done_ring, missed):
    assert reaches_a_missed_phase(ring, done_ring, 4 * done_ring) == missed
