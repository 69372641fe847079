"""Where the recurrent layer's two-pass form cuts few long chunks (kda_segments in wpp_api.cu), against a model of the launch: rounds
of preparation on all SMs for the first segment and beside the chain before it for the others."""
import ctypes
import math

import pytest

import paper_2609_35263_b200.binding as B

ROUND, BESIDE, START, GAP, STEP = 18.0, 20.0, 6.0, 12.0, 64 * 0.0525           # us, measured


def cut(requests, heads, tokens, sms=148):
    fn = B.load_library().wpp_kda_cut
    us, begin = ctypes.c_double(0), (ctypes.c_int32 * 16)()
    count = fn(ctypes.byref(B.KdaDesc(requests, heads, 128, 128, 0, 0, 0, 0, tokens)), sms, ctypes.byref(us), begin)
    return list(begin)[:count]


def model(begin, blocks, n, sms):
    """Total, and the longest that a chain waits for its preparation beyond the end of the chain before."""
    total, longest = math.ceil(begin[1] * n / (2 * sms)) * ROUND if len(begin) > 1 else math.ceil(blocks * n / (2 * sms)) * ROUND, 0.0
    for s in range(1, len(begin)):
        end = begin[s + 1] if s + 1 < len(begin) else blocks
        ready = math.ceil((end - begin[s]) * n / (2 * (sms - n))) * BESIDE + START
        busy = (begin[s] - begin[s - 1]) * STEP + GAP
        total += max(ready, busy)
        longest = max(longest, ready - busy)
    return total + (blocks - begin[-1]) * STEP, longest


def growing(blocks, n, sms):
    """Up to six segments that grow by the ratio of the two rates."""
    best = [0]
    growth = 0.0525 / (n * 0.9e-3 * 148 / (sms - n))
    if growth > 1.05:
        g = min(growth, 4.0)
        for s in range(2, 7):
            first = (g - 1) / (g ** s - 1) * blocks
            at = [int(first * (g ** i - 1) / (g - 1)) for i in range(s)]
            if first >= 4 and model(at, blocks, n, sms)[0] < model(best, blocks, n, sms)[0]:
                best = at
    return best


LENGTHS = sorted({int(2 ** (x / 4)) + d for x in range(24, 73) for d in (-1, 0, 37)})


@pytest.mark.parametrize("sms", [148, 132, 64, 8])
def test_cuts_cover_the_chunk_and_every_segment_but_the_last_has_room_for_its_state(sms):
    """A segment leaves its state where the operands of its last two blocks were."""
    counts = set()
    for n in list(range(1, 75)) + [148, 296]:
        for tokens in LENGTHS:
            begin = cut(1, n, tokens, sms)
            assert 1 <= len(begin) <= 16 and begin[0] == 0 and begin[-1] < tokens // 64 + 1
            assert all(b - a >= 2 for a, b in zip(begin, begin[1:])), (n, tokens, begin)
            counts.add(len(begin))
            assert cut(n, 1, tokens * n, sms) == begin               # chains: requests times heads
    assert sms == 8 or counts >= set(range(1, 10))


@pytest.mark.parametrize("sms", [148, 132])
def test_no_segment_but_the_first_is_waited_for(sms):
    """However long the chunk: within a round of preparation, and never slower than segments that just grow (with at most eight
    segments and eight rounds of the first one, the last preparation of 131,072 tokens x 32 heads was waited for 2.4 ms)."""
    for n in range(1, 42 * sms // 148):
        for tokens in LENGTHS:
            begin, blocks = cut(1, n, tokens, sms), tokens // 64 + 1
            total, wait = model(begin, blocks, n, sms)
            assert wait <= BESIDE, (n, tokens, begin, wait)
            assert total <= model(growing(blocks, n, sms), blocks, n, sms)[0] + 8 * max(0, len(begin) - 8) + 1e-6, (n, tokens, begin)


@pytest.mark.parametrize("tokens,heads,begin", [(16384, 32, [0, 37, 80, 130, 188]), (8192, 32, [0, 27, 56, 92]), (4096, 32, [0, 18, 39]),
                                                (2048, 32, [0, 18]), (12000, 16, [0, 18, 67]), (200, 32, [0]), (16384, 74, [0])])
def test_cuts_that_were_measured(tokens, heads, begin):
    assert cut(1, heads, tokens) == begin
