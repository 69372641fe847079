"""The recurrent layer's group form with its chains cut into pieces (wpp_kda_group.cu): who waits for whom, as a model of the
launch on the CPU."""
import os
import random
import re

import pytest

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
