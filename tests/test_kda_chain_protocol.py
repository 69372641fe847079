"""The hand-overs of the recurrent layer's chain kernel (wpp_kda_tc.cu) as a state machine, run through every interleaving.

A waiter on an mbarrier names a phase by its parity, so a barrier that completes twice while a waiter has seen neither looks
as if it had not completed at all.  The model has the issuing thread, the tensor pipe (which completes what was issued in
order, at any later time) and one thread of each row warpgroup; how many barriers the outputs have is read from the source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc", "wpp_kda_tc.cu")
STEPS = 5


def _programs(n_o):
    """Per thread: ("wait", barrier, phase), ("arrive", barrier) and ("issue", barrier that its completion arrives on)."""
    issuer, rows = [], {0: [], 1: []}
    for n in range(STEPS):
        if n >= 2:
            issuer.append(("wait", ("o_free", n & 1), n // 2 - 1))
        issuer += [("wait", ("shl", 0), n), ("issue", ("x", 0)), ("wait", ("uhl", 0), n), ("issue", ("s", 0)),
                   ("issue", ("o", n % n_o))]

    def outputs(n):
        return [("wait", ("o", n % n_o), n // n_o), ("arrive", ("o_free", n & 1))]

    for wg, prog in rows.items():
        for n in range(STEPS):
            if n:
                prog.append(("wait", ("s", 0), n - 1))
            prog += [("arrive", ("shl", 0)), ("wait", ("x", 0), n), ("arrive", ("uhl", 0))]
            if wg == 1 and n:
                prog += outputs(n - 1)
        if wg == 1:
            prog += outputs(STEPS - 1)
        prog.append(("wait", ("s", 0), STEPS - 1))
    return [issuer, rows[0], rows[1]]


ARRIVALS = {"shl": 2, "uhl": 2, "x": 1, "s": 1, "o": 1, "o_free": 1}


def _deadlock(n_o):
    """A reachable state in which nothing can run and not everything is done, or None."""
    progs = _programs(n_o)
    names = sorted({op[1] for p in progs for op in p})
    index = {b: i for i, b in enumerate(names)}
    start = ((0, 0, 0), (), tuple((0, 0) for _ in names))         # program counters, issued work, (phases, arrivals) per barrier
    seen, todo = {start}, [start]

    def arrive(bars, b):
        i = index[b]
        phases, count = bars[i]
        count += 1
        new = (phases + 1, 0) if count == ARRIVALS[b[0]] else (phases, count)
        return bars[:i] + (new,) + bars[i + 1:]

    while todo:
        pcs, pipe, bars = state = todo.pop()
        nexts = []
        if pipe:
            nexts.append((pcs, pipe[1:], arrive(bars, pipe[0])))
        for t, prog in enumerate(progs):
            if pcs[t] == len(prog):
                continue
            op = prog[pcs[t]]
            after = pcs[:t] + (pcs[t] + 1,) + pcs[t + 1:]
            if op[0] == "wait":
                if (bars[index[op[1]]][0] & 1) != (op[2] & 1):     # mbarrier.try_wait.parity
                    nexts.append((after, pipe, bars))
            elif op[0] == "arrive":
                nexts.append((after, pipe, arrive(bars, op[1])))
            else:
                nexts.append((after, pipe + (op[1],), bars))
        if not nexts and any(pc < len(p) for pc, p in zip(pcs, progs)):
            return state
        for s in nexts:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


def test_the_model_finds_the_wait_that_one_output_barrier_would_lose():
    assert _deadlock(1) is not None


def test_no_interleaving_of_the_chain_kernels_waits_blocks():
    src = open(SRC).read()
    chain = src[src.index("kda_tc_chain_kernel(const"):]
    n_o = len(set(re.findall(r"mbar_init\(bOReady(?:\((\d)\))?, 1\)", chain)))
    assert n_o in (1, 2)
    assert _deadlock(n_o) is None
