"""The word that the blocks of a peel meet on, across the 2^32nd arrival: its
low half counts arrivals and carries into the high half, which sums the
blocks' counts.  A model of the word (each block adds count << 32 | 1) against
what the library takes out of it at each meeting, with the sums small and
wrapping, arrivals below, at and past the carry."""
import pytest

import paper_2103_00154_gb300 as dsg


@pytest.mark.parametrize("wraps", [0, 1, 300])
@pytest.mark.parametrize("queued", [0, 12345, (1 << 32) - 9])
@pytest.mark.parametrize("blocks", [2, 152, 256, 304, 608])
def test_counts_across_the_carry(blocks, queued, wraps):
    count_of = dsg.lib().dsg_debug_meet_count
    M = 1 << 32
    # every block has arrived so often on each of the two words: 3 meetings short of a carry
    before = ((wraps + 1) * M // blocks - 3) * blocks
    words = [((queued << 32) + before) % (1 << 64)] * 2
    high, arrivals = [w >> 32 for w in words], [before] * 2
    carries = 0
    for meeting in range(14):
        par = meeting & 1
        handed = 0
        for b in range(blocks):
            count = (meeting * 7 + b) % 5
            words[par] = (words[par] + (count << 32) + 1) % (1 << 64)
            handed += count
        arrivals[par] += blocks
        carries += ((words[par] >> 32) - high[par]) % M != handed  # the plain difference is wrong
        assert count_of(words[par], high[par], arrivals[par] % M, blocks) == handed
        high[par] = words[par] >> 32
    assert carries == 2  # once on each word
