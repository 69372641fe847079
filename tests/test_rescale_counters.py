"""The counters from which the order of rescaling is chosen: every launch leaves its totals at its own end, whatever else runs; no
device memory is allocated for them, and contexts come and go beside a capture."""
import gc
import os
import re

import pytest
import torch

import paper_2609_35263_b200 as wpp

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc")


def test_a_context_allocates_no_device_memory_and_is_destroyed_without_a_cuda_call():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wpp_api.cu")).read())
    assert not re.search(r"cudaMalloc|cudaStreamCreate", src)
    destroy = src[src.index("int wpp_destroy("):src.index("int wpp_set_rescale_mode(")]
    assert "cuda" not in destroy


def test_the_shares_of_a_launch_pass_one_whole_number_and_only_with_its_last_cta():
    """The arithmetic of the kernel's end, for one launch at a time and for two that overlap in one slot."""
    def share(i, n):
        each = 0xffffffff // n
        return each if i else 2 ** 32 - each * (n - 1)

    ended = 12 << 32
    for n in (1, 2, 3, 7, 147, 148, 4096, 4095):
        for order in (range(n), reversed(range(n))):
            passed = []
            for i in order:
                passed.append(((ended & 0xffffffff) + share(i, n)) >> 32)
                ended += share(i, n)
            assert passed == [0] * (n - 1) + [1] and ended & 0xffffffff == 0
    a, b = [share(i, 148) for i in range(148)], [share(i, 3) for i in range(3)]
    for mix in (a[:100] + b + a[100:], b[:1] + a + b[1:], [x for p in zip(a[:3], b) for x in p] + a[3:]):
        passed = []
        for x in mix:
            passed.append(((ended & 0xffffffff) + x) >> 32)
            ended += x
        assert sum(passed) == 2 and passed[-1] == 1


def _wave(P, C, Hq, Hkv, ctas):
    import wpp_workloads as W
    from tests import gpu_harness as H

    w = W.custom_workload(P, C, Hq, Hkv, 128, 64, seed=61, spare_pages=2)
    g, d = H.device_inputs(w), H.desc_of(w)
    i32 = lambda a: torch.from_numpy(a.astype("int32")).cuda()
    bt, Pd, Cd = i32(w.block_tables), i32(w.prefix_lens), i32(w.chunk_lens)
    out = torch.empty_like(g["q"])

    def bind(c):
        plan = wpp.wpp_plan_tiles(c, d, w.prefix_lens, w.chunk_lens, opts=wpp.PlanOpts(256, 0, 1, ctas, 0, 1)).to_device()
        ws = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device="cuda")
        return lambda: wpp.wpp_prefill_attention_varlen(c, d, g["q"], out, None, g["k_pool"], g["v_pool"], bt, Pd, Cd, plan, workspace=ws)
    return bind


@pytest.mark.gpu
def test_a_launch_that_ends_beside_a_longer_one_has_left_its_totals():
    c = wpp.Context(0)
    long, short = _wave([100000], [4096], 1, 1, 1)(c), _wave([300], [200], 8, 2, 0)(c)
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    short(), long()                                       # (everything loaded)
    torch.cuda.synchronize()
    steps = []
    for call in (short, long):
        s0 = c.rescale_stats()[0]
        call()
        torch.cuda.synchronize()
        steps.append(c.rescale_stats()[0] - s0)
    assert steps[0] > 0 and steps[1] > 10 * steps[0]
    s0, _, _ = c.rescale_stats()
    with torch.cuda.stream(side):
        long()
        done = torch.cuda.Event()
        done.record()
    for i in range(1, 41):                                # (more launches than slots)
        with torch.cuda.stream(main):
            short()
        main.synchronize()
        assert not done.query(), "the long launch is over: nothing overlapped"
        # (one launch in sixteen has the long one's slot, and its totals may come with the next)
        assert c.rescale_stats()[0] - s0 >= (i - 1 if i % 16 == 0 else i) * steps[0]
    torch.cuda.synchronize()
    assert c.rescale_stats()[0] - s0 == 40 * steps[0] + steps[1]


@pytest.mark.gpu
def test_totals_never_fall_with_launches_on_two_streams():
    c = wpp.Context(0)
    calls = [_wave([500], [400], 4, 1, 60)(c), _wave([0, 90], [300, 10], 4, 1, 60)(c)]
    per = []
    for call in calls:
        s0 = c.rescale_stats()[0]
        call()
        torch.cuda.synchronize()
        per.append(c.rescale_stats()[0] - s0)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    s0, last = c.rescale_stats()[0], c.rescale_stats()[:2]
    for i in range(600):
        for call, stream in zip(calls, streams):
            with torch.cuda.stream(stream):
                call()
        now = c.rescale_stats()[:2]
        assert now[0] >= last[0] and now[1] >= last[1]
        last = now
    torch.cuda.synchronize()
    assert c.rescale_stats()[0] - s0 == 600 * sum(per)


@pytest.mark.gpu
def test_contexts_come_and_go():
    """More contexts than have counters, each with zero to begin with; the ones without launch all the same."""
    first = wpp.Context(0)
    bind = _wave([64], [100], 4, 1, 0)
    bind(first)()
    torch.cuda.synchronize()
    assert first.rescale_stats()[0] > 0
    first.close()
    many = [wpp.Context(0) for _ in range(260)]
    assert all(c.rescale_stats() == (0, 0, False) for c in many)
    bind(many[0])(), bind(many[-1])()
    torch.cuda.synchronize()
    assert many[0].rescale_stats()[0] > 0 and many[-1].rescale_stats()[0] == 0
    for c in many:
        c.close()


@pytest.mark.gpu
def test_contexts_are_created_and_destroyed_beside_a_capture():
    c, old = wpp.Context(0), wpp.Context(0)
    call = _wave([64], [100], 4, 1, 0)(c)
    call()
    torch.cuda.synchronize()
    s0 = c.rescale_stats()[0]
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    gc.disable()
    try:
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="global"):
            old.close()
            new = wpp.Context(0)
            call()
            new.close()
    finally:
        gc.enable()
    graph.replay()
    torch.cuda.synchronize()
    assert c.rescale_stats()[0] > s0
