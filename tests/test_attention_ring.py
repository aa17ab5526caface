"""The mma.sync attention kernel's ring of K and V tiles: who waits for which use of a slot.

Two groups of four warps take the tiles of a CTA in turn (even and odd ones) without a step in common, each warp waiting on
the mbarrier of a slot by the parity of the use it wants.  A parity names a use only to a waiter that has seen the use before
it: to one that has not, the barrier still open on use u - 1 looks like one that has completed use u.  So all uses of a slot
must belong to one group - TMA completions need not arrive in the order of the requests."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2606_12243_b200", "csrc", "attention_mma.cu")


def test_every_use_of_a_ring_slot_belongs_to_one_group_of_warps():
    ring = int(re.search(r"constexpr int RING = (\d+);", open(SRC).read()).group(1))
    group_of = {}                                              # slot -> the group that waits for it
    for tile in range(64):
        for request in (2 * tile, 2 * tile + 1):               # K and V of the tile, in the order of the requests
            assert group_of.setdefault(request % ring, tile & 1) == tile & 1, (ring, tile, request)


def test_a_parity_wait_that_skipped_a_use_returns_early():
    """The failing order, with the barrier as the hardware keeps it (a wait for parity p returns when the phase in progress
    has the other parity): tile 0's V is late, tile 1's K and V have landed and been read, tile 3's K shares its slot."""
    def passes(completed, use):
        return completed & 1 != use & 1                        # completed: uses that have landed, the phase in progress
    late = 0                                                   # slot 1 after request 1 (V of tile 0) has not landed yet
    assert passes(late, 1)                                     # request 6 = second use of slot 1 of 5: taken for landed
    assert not passes(late, 0) and not passes(1, 1)            # the group that waits for every use is held back
