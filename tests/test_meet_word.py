"""The word that the blocks of a peel meet on, across the 2^32nd arrival: its
low half counts arrivals and carries into the high half, which sums the
blocks' counts.  A model of the word (each block adds count << 32 | 1) against
the library's sum, with the words' sums small, at the carry and wrapping."""
import pytest

import paper_2103_00154_gb300 as dsg


@pytest.mark.parametrize("queued", [0, 12345, (1 << 32) - 9])
@pytest.mark.parametrize("blocks", [2, 152, 304, 608])
def test_sum_across_the_carry(blocks, queued):
    L = dsg.lib()
    per_word = (1 << 32) // blocks - 3  # arrivals of every block so far, on each of the two words
    words = [((queued << 32) + per_word * blocks) % (1 << 64)] * 2
    sums, arrivals = [queued, queued], [per_word * blocks] * 2
    carried = False
    for meeting in range(14):
        par = meeting & 1
        arrivals[par] += blocks
        for b in range(blocks):
            count = (meeting * 7 + b) % 5
            words[par] = (words[par] + (count << 32) + 1) % (1 << 64)
            sums[par] = (sums[par] + count) % (1 << 32)
        carried |= words[par] >> 32 != sums[par]
        assert L.dsg_debug_meet_sum(words[par], arrivals[par]) == sums[par]
    assert carried  # the plain high half is wrong here


def test_sum_in_the_longest_peel():
    arrivals = 608 << 31  # 2^31 rounds
    word = (arrivals + (77 << 32)) % (1 << 64)
    assert dsg.lib().dsg_debug_meet_sum(word, arrivals) == 77
