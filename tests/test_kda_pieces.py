"""The recurrent layer's group form with its chains cut into pieces (wpp_kda_group.cu): which waves are cut, and who waits for
whom, as a model of the launch on the CPU."""
import ctypes
import os
import random
import re

import pytest

import paper_2609_35263_b200.binding as B

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc")


def _kernel_source():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wpp_kda_group.cu")).read())
    return src[src.index("kda_group_kernel(const"):src.index("static int launch(")]


def _stuck(order, chains, pieces, sms, by_ticket):
    """CTAs of a launch started in `order` on `sms` SMs, a CTA each: whether pieces are left that can never run.  A CTA takes its
    piece from a counter as it starts, or from its own index; a piece holds its SM until the one before it has ended."""
    todo, on_sm, done, tickets = list(order), [], set(), iter(range(chains * pieces))
    while todo or on_sm:
        while todo and len(on_sm) < sms:
            cta = todo.pop(0)
            on_sm.append(next(tickets) if by_ticket else cta)
        over = [p for p in on_sm if p < chains or p - chains in done]
        if not over:
            return True
        done.update(over)
        on_sm = [p for p in on_sm if p not in done]
    return False


def _orders(n):
    rng = random.Random(n)
    yield list(range(n))
    yield list(range(n))[::-1]
    for _ in range(50):
        order = list(range(n))
        rng.shuffle(order)
        yield order


def test_the_model_finds_an_order_of_starting_in_which_pieces_by_index_wait_for_ever():
    assert any(_stuck(order, 20, 4, 16, by_ticket=False) for order in _orders(80))


def test_no_order_of_starting_leaves_a_piece_waiting():
    """CUDA does not say in which order the CTAs of a grid start."""
    body = _kernel_source()
    by_ticket = re.search(r"piece\s*=\s*\*ticket\s*/", body) is not None and "blockIdx.z" not in body
    for chains, pieces, sms in ((20, 4, 16), (16, 8, 16), (37, 2, 5)):
        for order in _orders(chains * pieces):
            assert not _stuck(order, chains, pieces, sms, by_ticket)


def _limits_until_the_end(pieces, failure_is_told):
    """How many limits of a wait pass, one after the other, until the pieces of a chain have ended whose first one gave up."""
    limits, told = 1, failure_is_told
    for _ in range(pieces - 1):
        if not told:
            limits += 1
    return limits


def test_the_pieces_behind_one_that_gave_up_do_not_wait_for_their_limits():
    """Half a second each: eight pieces in fourteen rounds of CTAs would keep the GPU for minutes."""
    body = _kernel_source()
    told = re.search(r"st_release\(seen, dead \? -1 :", body) is not None and re.search(r"if \(at < 0 \|\|", body) is not None
    assert _limits_until_the_end(8, False) == 8
    assert _limits_until_the_end(8, told) == 1


def choice(requests, heads, tokens, sms=148):
    """(form, pieces, longest chunk) that the library chooses for layout 0; form 1 is the one that is cut."""
    fn = B.load_library().wpp_kda_choice
    fn.argtypes = [ctypes.POINTER(B.KdaDesc), ctypes.c_int, ctypes.POINTER(ctypes.c_int64), ctypes.POINTER(ctypes.c_int)]
    longest, pieces = ctypes.c_int64(0), ctypes.c_int(0)
    form = fn(ctypes.byref(B.KdaDesc(requests, heads, 128, 128, 0, 0, 0, 0, tokens)), sms, ctypes.byref(longest), ctypes.byref(pieces))
    return form, pieces.value, longest.value


@pytest.mark.parametrize("lens,heads", [([166] * 4 + [22], 32), ([186] * 4 + [93, 19], 32), ([130] * 5, 32), ([190] * 5, 32)])
def test_short_chains_are_not_cut(lens, heads):
    """Cut in two, the first wave takes 53 us and not 45, the second 67 and not 59."""
    assert choice(len(lens), heads, sum(lens))[:2] == (1, 1)


def test_a_piece_has_96_tokens_and_its_chains_fill_the_sms():
    seen = set()
    for sms in (148, 132, 64):
        for heads in (1, 7, 8, 16, 32, 64, 300):
            for requests in (1, 2, 5, 6, 8, 13, 20, 64):
                for mean in (64, 100, 150, 191, 192, 250, 400, 1000, 2048, 5000):
                    form, pieces, longest = choice(requests, heads, requests * mean, sms)
                    assert 1 <= pieces <= 8
                    if pieces > 1:
                        seen.add(pieces)
                        assert form == 1 and requests * heads >= sms and mean >= 96 * pieces
                        assert requests == 1 or longest >= mean
    assert seen >= {2, 3, 4, 5}


@pytest.mark.parametrize("requests,heads,mean,pieces", [(8, 32, 2048, 4), (6, 32, 2048, 3), (5, 32, 1000, 5), (20, 8, 800, 4), (64, 32, 256, 1),
                                                        (5, 32, 256, 2), (8, 32, 1024, 1)])
def test_waves_whose_cut_was_measured(requests, heads, mean, pieces):
    assert choice(requests, heads, requests * mean)[:2] == (1, pieces)
