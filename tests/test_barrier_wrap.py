"""The depletion's grid barrier counts arrivals over all barriers of a call.  A long chain of
rounds (one photon in tens of millions of hits) takes the 32-bit counter past its end: a block
must neither leave before the last block arrives nor wait for ever.  No GPU is needed."""
import pytest

from paper_1608_01125_gb300 import binding

M = 1 << 32


@pytest.mark.parametrize("blocks", [1, 2, 3, 19, 152, 1024])
@pytest.mark.parametrize("start", [1, M - 5000, M - 1, 2 * M - 1025, 7 * M // 2])
def test_a_block_leaves_exactly_when_all_have_arrived(blocks, start):
    import __graft_entry__
    __graft_entry__.build()
    arrived = binding.lib().trilens_debug_arrived
    first = start // blocks
    for done in range(first, first + 12):  # the barriers around the wrap
        want = done * blocks
        # a block that waits is between its own arrival and the next barrier's end
        for have in {want - blocks + 1, want - blocks + blocks // 2 + 1, want - 1, want, want + 1,
                     want + blocks - 1}:
            if have >= want - blocks + 1:
                assert arrived(have % M, want % M) == (have >= want), (done, have - want)
