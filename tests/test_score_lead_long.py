"""The chunk length of the two-pass score kernel at long sequences: the lead that completing a head needs
must fit the ring of chunk records, on both sides of every line where the rule lengthens the chunks.  The
limits are read from the source; the schedule is the model of test_score_lead.py."""
import os
import re

import pytest

from tests.test_score_lead import MAX_LEAD_CHUNKS, RING, TILE, ceil_div, run

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_09754_b200", "csrc",
                   "score_sm100.cu")
SMS = 148


def _constant(name):
    return int(re.search(r"constexpr int %s = (\d+);" % name, open(SRC).read()).group(1))


def _chunk_tiles(n, split, wanted):
    """The kernel's rule: what is wanted, but at most (kMaxLeadChunks - 1) rounds of CTAs per head."""
    most = (_constant("kMaxLeadChunks") - 1) * SMS >> split
    return max(wanted, ceil_div(ceil_div(n, TILE), most))


def test_the_model_has_the_limits_of_the_source():
    assert (_constant("kMaxLeadChunks"), _constant("kRing"), _constant("kTile")) == (MAX_LEAD_CHUNKS, RING, TILE)
    text = open(SRC).read()
    assert "(kMaxLeadChunks - 1) * sms >> split" in text and "return wanted > least ? wanted : least;" in text


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("wanted", [1, 4, 8])
@pytest.mark.parametrize("factor", [0.5, 1.0, 1.01, 1.1, 1.6, 2.5])
def test_every_wait_ends_at_long_sequences(split, wanted, factor):
    n = int(factor * ((MAX_LEAD_CHUNKS - 1) * SMS >> split) * wanted * TILE)
    for heads, radius in ((1, 3), (2, 31)):
        assert run([n], 1, heads, split, 32, radius, _chunk_tiles(n, split, wanted), SMS, extra=12)


def test_chunks_as_short_as_wanted_stall_there():
    assert not run([1200000], 1, 1, 1, 32, 3, 8, SMS, 12)
    assert run([1200000], 1, 1, 1, 32, 3, _chunk_tiles(1200000, 1, 8), SMS, 12)


@pytest.mark.parametrize("wanted,extra", [(12, 12), (16, 12), (16, 20)])
@pytest.mark.parametrize("factor", [0.5, 1.0, 1.01, 1.6])
def test_every_wait_ends_with_the_chunks_of_split_groups(wanted, extra, factor):
    n = int(factor * ((MAX_LEAD_CHUNKS - 1) * SMS >> 1) * wanted * TILE)
    for heads, radius in ((1, 3), (2, 31)):
        assert run([n], 1, heads, 1, 32, radius, _chunk_tiles(n, 1, wanted), SMS, extra)
    for lens in ([8193], [32768, 100], [32769, 9000], [131072], [151552], [151553]):
        assert run(lens, 2, 4, 1, 32, 3, _chunk_tiles(max(lens), 1, wanted), SMS, extra)
