"""wpp_kda_chunk (CUDA, through the C ABI) against the fp64 oracle of the recurrent-state layer (Section 3.1 update,
Section 3.2 snapshots), element by element on seeded inputs, plus the properties that hold at any size.

Tolerances: the token-by-token forms (layouts 1, 2) compute in fp32 (relative error of a step about 1e-7, a few
1e-6 after thousands of contracting steps); the chunk-parallel tensor-core form (layout 3) multiplies operands of
16 significant bits (two bf16 terms each, relative 2^-17 per factor) and accumulates in fp32, so a product of 64 or
128 terms carries about 1e-5 of its typical term; all forms round outputs to bf16 (relative 2^-9), states stay fp32.
  outputs : |delta| <= 2^-8 |ref| + 1e-4 max|ref|          states : |delta| <= 1e-4 max|ref|"""
import numpy as np
import pytest
import torch

import paper_2609_35263_b200 as wpp
import wpp_workloads as W
from oracle import kda as O
from tests import gpu_harness as H
from tests.test_kda_pieces import choice
from tests.test_kda_segments import cut

pytestmark = pytest.mark.gpu


def _oracle(w, t, heads=None):
    hs = slice(None) if heads is None else heads
    f = lambda x: x[:, hs].double().numpy()
    pool = t["state_pool"][:, hs].double().numpy().copy()
    o = O.kda_chunk(f(t["q"]), f(t["k"]), f(t["v"]), f(t["alpha"]), f(t["beta"]), w.chunk_lens, pool, w.state_in,
                    w.state_out, w.prefix_lens, w.snap_interval, w.snap_slots)
    return o, pool


def _gpu(w, t, state_in=None, state_out=None, layout=0):
    dev = torch.device("cuda")
    d = {k: v.to(dev) for k, v in t.items()}
    i32 = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    T, Hh = int(t["q"].shape[0]), int(t["q"].shape[1])
    ws = torch.full((wpp.wpp_kda_workspace_bytes(len(w.chunk_lens), Hh, T),), 0xFF, dtype=torch.uint8, device=dev)
    out = wpp.wpp_kda_chunk(H.ctx(), d["q"], d["k"], d["v"], d["alpha"], d["beta"],
                            torch.from_numpy(w.row_offsets).to(dev), d["state_pool"],
                            i32(w.state_in if state_in is None else state_in),
                            i32(w.state_out if state_out is None else state_out),
                            prefix_lens=i32(w.prefix_lens), snap_interval=w.snap_interval,
                            snap_slots=i32(w.snap_slots), status=status, layout=layout, workspace=ws)
    torch.cuda.synchronize()
    return out.float().cpu().double().numpy(), d["state_pool"].cpu().double().numpy(), int(status.item())


def _close_out(got, ref, what):
    if ref.size == 0:
        return
    bound = 2.0 ** -8 * np.abs(ref) + 1e-4 * np.abs(ref).max()
    bad = np.abs(got - ref) > bound
    assert not bad.any(), f"{what}: {bad.sum()} outputs off, worst {np.abs(got - ref).max():.3e}"


def _close_state(got, ref, what):
    assert np.abs(got - ref).max() <= 1e-4 * max(np.abs(ref).max(), 1e-30), f"{what}: {np.abs(got - ref).max():.3e}"


@pytest.mark.parametrize("lens,prefix,interval,H_", [
    ([37, 5, 64, 0, 1, 16, 17, 130], [11, 0, 128, 7, 0, 16, 3, 1000], 16, 2),     # ragged, stage tails, empty chunk
    ([300], [0], 0, 3),                                                            # one request from the zero state
    ([15, 16, 17, 31, 32, 33], [1, 2, 3, 4, 5, 6], 7, 1),                          # around the staging size; odd interval
])
@pytest.mark.parametrize("layout", [1, 2, 3])       # one CTA per (request, head) / four column slices / chunk-parallel
def test_ragged_batches_match_the_oracle(lens, prefix, interval, H_, layout):
    w = W.kda_workload("ragged", 11, lens, H_, prefix, snap_interval=interval)
    t = w.tensors()
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=layout)
    assert status == 0
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")
    # slots nobody writes keep their bits
    written = set(int(s) for s in w.state_out if s >= 0)
    if w.snap_slots is not None:
        written |= set(int(s) for s in w.snap_slots.ravel() if s >= 0)
    for s in range(w.num_slots):
        if s not in written:
            assert np.array_equal(got_pool[s], t["state_pool"][s].double().numpy())


@pytest.mark.parametrize("layout", [1, 2, 3])
def test_a_long_chain_stays_within_tolerance(layout):
    w = W.kda_workload("long", 5, [2048], 1, [4096])
    t = w.tensors()
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=layout)
    assert status == 0
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")


@pytest.mark.parametrize("layout,cut", [(1, (64, 32)), (1, (37, 20)), (2, (64, 32)), (2, (37, 20)), (3, (59, 64))])
def test_splitting_a_chunk_and_resuming_is_bit_identical(layout, cut):
    """Section 3.2: the state after exactly r tokens is all a recurrent layer needs.  The token-by-token forms'
    arithmetic per token does not depend on where a chunk starts, so one call and two resumed calls agree to the bit
    for any cut; the chunk-parallel form works on blocks of 64 sequence positions, so it does for cuts at multiples
    of 64 (request 0 has 5 cached tokens: its cut after 59 tokens is position 64)."""
    w = W.kda_workload("whole", 3, [100, 64], 2, [5, 0], resume=[True, False])
    t = w.tensors()
    whole_o, whole_pool, _ = _gpu(w, t, layout=layout)
    rows = w.row_offsets
    parts_o = np.zeros_like(whole_o)
    pool = t["state_pool"].clone()
    for first in (True, False):
        lens = [cut[i] if first else int(w.chunk_lens[i]) - cut[i] for i in range(2)]
        sel = np.concatenate([np.arange(rows[i] + (0 if first else cut[i]), rows[i] + (cut[i] if first else w.chunk_lens[i]))
                              for i in range(2)])
        wp = W.kda_workload("part", 3, lens, 2, [5, 0] if first else [5 + cut[0], cut[1]])
        wp.num_slots = w.num_slots
        tp = {k: (v[sel].contiguous() if k != "state_pool" else pool) for k, v in t.items()}
        s_in = w.state_in if first else w.state_out          # the second call resumes from what the first stored
        o, new_pool, status = _gpu(wp, tp, state_in=s_in, state_out=w.state_out, layout=layout)
        assert status == 0
        parts_o[sel] = o
        pool = torch.from_numpy(new_pool).float()
    assert np.array_equal(parts_o, whole_o)
    assert np.array_equal(pool.double().numpy(), whole_pool)


def test_splitting_inside_a_block_stays_within_tolerance_in_the_chunk_parallel_form():
    """A cut that is not a multiple of 64 moves a block boundary of the chunk-parallel form: the two resumed calls
    then round differently from the single call, and both stay within the tolerances against the oracle."""
    w = W.kda_workload("whole", 3, [100, 64], 2, [5, 0], resume=[True, False])
    t = w.tensors()
    ref_o, ref_pool = _oracle(w, t)
    rows, cut = w.row_offsets, (37, 20)
    parts_o = np.zeros_like(ref_o)
    pool = t["state_pool"].clone()
    for first in (True, False):
        lens = [cut[i] if first else int(w.chunk_lens[i]) - cut[i] for i in range(2)]
        sel = np.concatenate([np.arange(rows[i] + (0 if first else cut[i]), rows[i] + (cut[i] if first else w.chunk_lens[i]))
                              for i in range(2)])
        wp = W.kda_workload("part", 3, lens, 2, [5, 0] if first else [5 + cut[0], cut[1]])
        wp.num_slots = w.num_slots
        tp = {k: (v[sel].contiguous() if k != "state_pool" else pool) for k, v in t.items()}
        o, new_pool, status = _gpu(wp, tp, state_in=w.state_in if first else w.state_out, state_out=w.state_out, layout=3)
        assert status == 0
        parts_o[sel] = o
        pool = torch.from_numpy(new_pool).float()
    _close_out(parts_o, ref_o, "outputs of the two resumed calls")
    for i in range(2):
        _close_state(pool[w.state_out[i]].double().numpy(), ref_pool[w.state_out[i]], "final state")


@pytest.mark.parametrize("layout", [1, 2, 3])
def test_tiny_and_zero_decays(layout):
    """Decays of exactly 0 (a channel forgets everything), of 1e-6 and 1e-20, and runs of small ones."""
    w = W.kda_workload("decays", 17, [90, 40], 2, [3, 0])
    t = w.tensors()
    rng = np.random.default_rng(17)
    a = t["alpha"].numpy()
    T = a.shape[0]
    for val, count in ((0.0, 40), (1e-6, 40), (1e-20, 20), (0.3, 2000)):
        idx = (rng.integers(0, T, count), rng.integers(0, 2, count), rng.integers(0, 128, count))
        a[idx] = val
    a[50:58, 0, 7] = 0.05                                      # eight small decays in a row on one channel
    a[0, :, :] = 0.0                                           # the first token forgets the resumed state entirely
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=layout)
    assert status == 0 and np.isfinite(got_o).all() and np.isfinite(got_pool).all()
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")


@pytest.mark.parametrize("layout", [1, 2, 3])
def test_in_place_slots_and_pure_decay(layout):
    # state_out == state_in updates a slot in place; with beta = 0 and alpha = 1 the state must not change at all
    w = W.kda_workload("inplace", 9, [50, 20], 2, [10, 10])
    t = w.tensors()
    t["beta"].zero_()
    t["alpha"].fill_(1.0)
    got_o, got_pool, status = _gpu(w, t, state_out=w.state_in, layout=layout)
    assert status == 0
    assert np.array_equal(got_pool, t["state_pool"].double().numpy())
    ref = np.einsum("rhkv,rhk->rhv", t["state_pool"][[0] * 50 + [1] * 20].double().numpy(), t["q"].double().numpy())
    _close_out(got_o, ref, "o = S0^T q")


@pytest.mark.parametrize("layout,requests,heads", [(1, 23, 29), (1, 149, 1), (2, 23, 8)])
def test_more_items_than_sms_are_taken_over_one_after_the_other(layout, requests, heads):
    """The token-by-token forms' CTAs go on with items that no CTA has started: lengths on both sides of a stage of 16 tokens and
    of the 8 left when the next item is asked for, empty chunks, requests from the zero state and without a final state."""
    rng = np.random.default_rng(requests)
    lens = [int(n) for n in rng.choice([0, 1, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32, 33, 40], requests)]
    w = W.kda_workload("items", 5, lens, heads, [int(n) for n in rng.integers(0, 40, requests)], snap_interval=13)
    t = w.tensors()
    w.state_in[rng.random(requests) < 0.2] = -1
    w.state_out[rng.random(requests) < 0.2] = -1
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=layout)
    assert status == 0
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")


def test_bad_slot_ids_are_reported_and_skipped():
    w = W.kda_workload("bad", 2, [20, 20, 20], 1, [4, 4, 4])
    t = w.tensors()
    s_in, s_out = w.state_in.copy(), w.state_out.copy()
    s_in[1], s_out[2] = w.num_slots + 5, -7
    got_o, got_pool, status = _gpu(w, t, state_in=s_in, state_out=s_out)
    assert status == 3                                                 # WPP_ERR_BOUNDS
    w.state_in, w.state_out = np.where(s_in >= w.num_slots, -1, s_in), np.where(s_out < -1, -1, s_out)
    ref_o, ref_pool = _oracle(w, t)                                    # bad ids behave like -1
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")


def test_argument_errors():
    dev = torch.device("cuda")
    z = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device=dev)
    ro = torch.tensor([0, 4], dtype=torch.int64, device=dev)
    slot = torch.zeros(1, dtype=torch.int32, device=dev)
    pool = z(1, 1, 64, 64, dt=torch.float32)
    with pytest.raises(wpp.WppError) as e:                            # d_k = d_v = 64 is not built
        wpp.wpp_kda_chunk(H.ctx(), z(4, 1, 64), z(4, 1, 64), z(4, 1, 64), z(4, 1, 64, dt=torch.float32),
                          z(4, 1, dt=torch.float32), ro, pool, slot, slot)
    assert e.value.status == 2
    pool = z(1, 1, 128, 128, dt=torch.float32)
    with pytest.raises(wpp.WppError) as e:                            # no such layout
        wpp.wpp_kda_chunk(H.ctx(), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128, dt=torch.float32),
                          z(4, 1, dt=torch.float32), ro, pool, slot, slot, layout=4)
    assert e.value.status == 1
    with pytest.raises(wpp.WppError) as e:                            # the chunk-parallel form needs its workspace
        wpp.wpp_kda_chunk(H.ctx(), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128, dt=torch.float32),
                          z(4, 1, dt=torch.float32), ro, pool, slot, slot, layout=3)
    assert e.value.status == 5
    small = torch.empty(1024, dtype=torch.uint8, device=dev)
    with pytest.raises(wpp.WppError) as e:
        wpp.wpp_kda_chunk(H.ctx(), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128, dt=torch.float32),
                          z(4, 1, dt=torch.float32), ro, pool, slot, slot, layout=3, workspace=small)
    assert e.value.status == 5
    assert wpp.wpp_kda_workspace_bytes(1, 1, 4) > 1024
    with pytest.raises(wpp.WppError) as e:                            # periodic snapshots need prefix_lens
        wpp.wpp_kda_chunk(H.ctx(), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128), z(4, 1, 128, dt=torch.float32),
                          z(4, 1, dt=torch.float32), ro, pool, slot, slot, snap_interval=2,
                          snap_slots=torch.zeros(1, 2, dtype=torch.int32, device=dev))
    assert e.value.status == 1


@pytest.mark.parametrize("lanes,chunk", [(8, 2048), (1, 16384)])
def test_full_size_wave_on_sampled_heads(lanes, chunk):
    """The benchmark's waves (8 lanes x 2,048 tokens: one CTA per pair; one lane x 16,384 tokens: the library picks
    four column slices per pair), 32 heads, resumed states: the oracle recomputes sampled (request, head) chains and
    all of their outputs and final states are compared."""
    w = W.kda_wave(lanes, chunk)
    t = w.tensors()
    got_o, got_pool, status = _gpu(w, t)
    assert status == 0
    rows = w.row_offsets
    for req, head in (((0, 0), (3, 17), (7, 31)) if lanes == 8 else ((0, 5),)):
        sl = slice(rows[req], rows[req + 1])
        sub = W.kda_workload("one", 0, [int(w.chunk_lens[req])], 1, [int(w.prefix_lens[req])])
        sub.num_slots, sub.state_in, sub.state_out = w.num_slots, w.state_in[req:req + 1], w.state_out[req:req + 1]
        ts = {k: (v[sl] if k != "state_pool" else v) for k, v in t.items()}
        ref_o, ref_pool = _oracle(sub, ts, heads=slice(head, head + 1))
        _close_out(got_o[sl, head:head + 1], ref_o, f"outputs of request {req} head {head}")
        _close_state(got_pool[w.state_out[req], head], ref_pool[w.state_out[req], 0], "final state")


@pytest.mark.parametrize("seed", range(24))
def test_random_waves_in_the_chunk_parallel_form(seed):
    """Seeded random waves for the chunk-parallel form: chunk lengths around the block size, prefixes at every
    alignment, snapshot intervals from 1 (every token is a sub-block of its own) to beyond a block, some channels with
    zero and tiny decays (extra cuts), odd head counts, resumed and zero states - all against the oracle."""
    rng = np.random.default_rng(4000 + seed)
    R = int(rng.integers(1, 6))
    H_ = int(rng.choice([1, 2, 3]))
    lens = [int(x) for x in rng.choice([0, 1, 2, 31, 63, 64, 65, 100, 127, 128, 129, 200, 333], R)]
    if sum(lens) == 0:
        lens[0] = 70
    prefix = [int(x) for x in rng.choice([0, 1, 5, 63, 64, 65, 100, 128, 1000, 4097], R)]
    interval = int(rng.choice([0, 0, 1, 2, 3, 16, 50, 64, 65, 200]))
    w = W.kda_workload("fuzz", 100 + seed, lens, H_, prefix, resume=rng.random(R) < 0.7, snap_interval=interval)
    t = w.tensors()
    if seed % 3 == 0 and w.total_tokens > 0:
        a = t["alpha"].numpy()
        T = a.shape[0]
        for val, count in ((0.0, 6), (1e-9, 6), (1e-30, 4), (0.2, 200)):
            idx = (rng.integers(0, T, count), rng.integers(0, H_, count), rng.integers(0, 128, count))
            a[idx] = val
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=3)
    assert status == 0 and np.isfinite(got_o).all() and np.isfinite(got_pool).all()
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")


@pytest.mark.parametrize("H_", [1, 7, 9, 17])        # 5 requests, with CTAs of 32 columns (up to 37 chains), of 64 (up to 74), of 128
@pytest.mark.parametrize("interval,decays", [(0, False), (7, True), (64, False), (1000, True)])
def test_groups_of_sixteen_positions_match_the_oracle(H_, interval, decays):
    """The library's choice for short chunks, groups of 16 positions with the state in registers: chunk lengths and
    prefixes around the group size, an empty chunk, snapshots inside groups, decays that have to end a group or go to
    the state directly.  Operands have 16 significant bits as in the chunk-parallel form: the same tolerances.  (One chunk is
    nearly four times the mean: a wave that is left to the two passes for it has to come out the same.  Which form ran is
    checked by test_the_group_form_matches_the_oracle_and_is_the_one_that_ran.)"""
    lens, prefix = [0, 1, 17, 130, 333], [5, 16, 31, 0, 4097]
    w = W.kda_workload("groups", 70 + H_, lens, H_, prefix, resume=[True, False, True, False, True], snap_interval=interval)
    t = w.tensors()
    if decays:
        rng = np.random.default_rng(H_)
        a = t["alpha"].numpy()
        for val, count in ((0.0, 6), (1e-9, 6), (1e-30, 4), (0.2, 200)):
            a[rng.integers(0, a.shape[0], count), rng.integers(0, H_, count), rng.integers(0, 128, count)] = val
    got_o, got_pool, status = _gpu(w, t)
    assert status == 0
    heads = [0, H_ - 1]
    ref_o, ref_pool = _oracle(w, t, heads=heads)
    _close_out(got_o[:, heads], ref_o, "outputs")
    _close_state(got_pool[:, heads], ref_pool, "state pool")


@pytest.mark.parametrize("lens,prefix,interval", [([5000], [70], 0), ([9000], [0], 192), ([14000, 10, 0], [63, 5, 64], 1000),
                                                  ([4500, 4200], [0, 129], 64)])
def test_long_chunks_in_segments_match_the_oracle(lens, prefix, interval):
    """Few long chains run the chunk-parallel form in segments, the preparation of one beside the chain of the one before,
    the state handed from chain to chain: requests of unequal length (some end in the first segment), snapshots on and
    off the cuts.  The arithmetic is that of one piece: the same tolerances, and the same bits as two resumed calls cut
    at a multiple of 64 positions."""
    w = W.kda_workload("segments", 91, lens, 2, prefix, snap_interval=interval)
    t = w.tensors()
    ref_o, ref_pool = _oracle(w, t)
    got_o, got_pool, status = _gpu(w, t, layout=3)
    assert status == 0
    _close_out(got_o, ref_o, "outputs")
    _close_state(got_pool, ref_pool, "state pool")
    if len(lens) == 1 and interval == 0:
        cut = 64 * 20 - prefix[0] % 64
        pool, parts = t["state_pool"].clone(), []
        for sl, s_in, pre in ((slice(0, cut), w.state_in, prefix[0]), (slice(cut, lens[0]), w.state_out, prefix[0] + cut)):
            wp = W.kda_workload("part", 91, [sl.stop - sl.start], 2, [pre])
            wp.num_slots = w.num_slots
            o, new_pool, status = _gpu(wp, {k: (v[sl].contiguous() if k != "state_pool" else pool) for k, v in t.items()},
                                       state_in=s_in, state_out=w.state_out, layout=3)
            assert status == 0
            parts.append(o)
            pool = torch.from_numpy(new_pool).float()
        assert np.array_equal(np.concatenate(parts), got_o)
        assert np.array_equal(pool.double().numpy(), got_pool)


@pytest.mark.parametrize("lens,prefix,interval,H_,segments", [([4096], [70], 0, 32, 3), ([4096], [0], 1152, 32, 3), ([4100], [129], 1000, 32, 3),
                                                              ([4500, 3692], [63, 0], 640, 16, 3), ([9000, 10, 0], [0, 5, 64], 1000, 11, 3),
                                                              ([16384], [0], 4096, 32, 5)])
def test_three_segments_and_more_match_the_oracle(lens, prefix, interval, H_, segments):
    """As above with chains enough for more than a few segments: how many ran is asserted, and snapshots lie on the cuts (block 18
    of 64 tokens: 1,152) and off them."""
    assert len(cut(len(lens), H_, sum(lens))) == segments
    w = W.kda_workload("segments", 92, lens, H_, prefix, snap_interval=interval)
    t = w.tensors()
    launches = H.ctx().launch_count()
    got_o, got_pool, status = _gpu(w, t, layout=3)
    assert status == 0 and H.ctx().launch_count() - launches == 1 + 2 * segments
    heads = [0, H_ - 1]
    ref_o, ref_pool = _oracle(w, t, heads=heads)
    _close_out(got_o[:, heads], ref_o, "outputs")
    _close_state(got_pool[:, heads], ref_pool, "state pool")


@pytest.mark.parametrize("tokens,H_,at_least", [(16384, 32, 5), (32768, 40, 9)])
def test_any_number_of_segments_has_the_bits_of_two_resumed_calls(tokens, H_, at_least):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(tokens)
    normal = lambda *shape: torch.empty(*shape, device=dev).normal_(generator=g)
    q, k, v = (normal(tokens, H_, 128).mul_(f).bfloat16() for f in (0.088, 0.088, 1.0))
    alpha, beta = torch.sigmoid(normal(tokens, H_, 128) + 4.0), torch.sigmoid(normal(tokens, H_))
    start = normal(2, H_, 128, 128).mul_(0.1)
    status, i32 = torch.zeros(1, dtype=torch.int32, device=dev), lambda *x: torch.tensor(x, dtype=torch.int32, device=dev)

    def run(pool, lo, hi, s_in):
        n, launches = hi - lo, H.ctx().launch_count()
        ws = torch.full((wpp.wpp_kda_workspace_bytes(1, H_, n),), 0xFF, dtype=torch.uint8, device=dev)
        out = wpp.wpp_kda_chunk(H.ctx(), q[lo:hi], k[lo:hi], v[lo:hi], alpha[lo:hi], beta[lo:hi],
                                torch.tensor([0, n], dtype=torch.int64, device=dev), pool, i32(s_in), i32(1), prefix_lens=i32(lo),
                                status=status, layout=3, workspace=ws)
        segments = (H.ctx().launch_count() - launches - 1) // 2
        assert segments == len(cut(1, H_, n))
        return out, segments

    whole, parts = start.clone(), start.clone()
    out, segments = run(whole, 0, tokens, 0)
    assert segments >= at_least
    middle = tokens // 3 // 64 * 64
    first, second = run(parts, 0, middle, 0)[0], run(parts, middle, tokens, 1)[0]
    assert int(status.item()) == 0
    assert torch.equal(torch.cat([first, second]).view(torch.int16), out.view(torch.int16)) and torch.equal(parts, whole)


def test_calls_of_few_long_chains_end_alike_however_cold_the_caches_are():
    """Few long chains start the chain kernel six times a call, beside a preparation that fills the memory system: three
    hundred calls, each from an idle device with its caches overwritten, end without a wait that ran out and with one
    result."""
    w = W.kda_workload("cold", 97, [6000], 8, [128])
    t = w.tensors()
    dev = torch.device("cuda")
    d = {k: v.to(dev) for k, v in t.items()}
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)
    rows, s_in, s_out, prefix = torch.from_numpy(w.row_offsets).to(dev), i32(w.state_in), i32(w.state_out), i32(w.prefix_lens)
    ws = torch.empty(wpp.wpp_kda_workspace_bytes(1, 8, 6000), dtype=torch.uint8, device=dev)
    cold = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    out, bad, first = torch.empty_like(d["v"]), torch.zeros(1, dtype=torch.int64, device=dev), None
    launches = H.ctx().launch_count()
    for i in range(300):
        cold.fill_(i & 1)
        torch.cuda.synchronize()
        wpp.wpp_kda_chunk(H.ctx(), d["q"], d["k"], d["v"], d["alpha"], d["beta"], rows, d["state_pool"], s_in, s_out, out=out,
                          prefix_lens=prefix, status=status, layout=3, workspace=ws)
        if first is None:
            first = out.clone()
        bad += (out.view(torch.int16) != first.view(torch.int16)).any()
    assert int(status.item()) == 0 and int(bad.item()) == 0
    assert H.ctx().launch_count() - launches > 300 * 3                 # in segments


@pytest.mark.parametrize("layout", [0, 1, 2, 3])
@pytest.mark.parametrize("C,interval", [(33, 32), (65, 64), (100, 7)])
def test_a_snapshot_slot_may_be_the_slot_of_the_chunk_end(layout, C, interval):
    """A request's periodic snapshots may go to the slot that its state at the chunk end goes to (no other request's slot):
    the last one written is the state at the end, however soon after the snapshot it follows and whichever way either is
    stored."""
    R, H_ = 40, 4
    w = W.kda_workload("same slot", 53, [C] * R, H_, [0] * R, snap_interval=interval)
    w.snap_slots[:] = w.state_out[:, None]
    t = w.tensors()
    heads = [0, H_ - 1]
    _, ref_pool = _oracle(w, t, heads=heads)
    for _ in range(5):
        _, got_pool, status = _gpu(w, t, layout=layout)
        assert status == 0
        _close_state(got_pool[:, heads], ref_pool, "state pool")


@pytest.mark.parametrize("shift", [None, 8.0, 1.0])                     # decays: the workload's, long memory, short memory
@pytest.mark.parametrize("H_", [9, 17, 33])                             # CTAs of 32, 64 and 128 columns
def test_groups_of_sixteen_positions_are_no_further_from_64_bits_than_the_two_passes(H_, shift):
    """What the library chooses for 4 x 192 tokens against the form that it stands in for (layout 3): the root mean square
    error of the states against 64 bits is no larger.  That the choice was the group form shows in the states' last bits."""
    w = W.kda_workload("error", 60 + H_, [192] * 4, H_, [0, 64, 5, 100])
    t = w.tensors()
    if shift is not None:
        g = torch.Generator().manual_seed(H_)
        t["alpha"] = torch.sigmoid(shift + 2 * torch.randn(t["alpha"].shape, generator=g))
    heads = [0, H_ - 1]
    _, ref_pool = _oracle(w, t, heads=heads)
    err, pools = [], []
    for layout in (0, 3):
        _, pool, status = _gpu(w, t, layout=layout)
        assert status == 0
        pools.append(pool)
        err.append(np.sqrt(np.mean((pool[w.state_out][:, heads] - ref_pool[w.state_out]) ** 2)))
    assert not np.array_equal(pools[0], pools[1])
    assert err[0] <= err[1], err


@pytest.mark.parametrize("H_", [1, 7, 17, 30])       # 6 requests: CTAs of 32 columns, of 64, of 128, and two rounds of them
@pytest.mark.parametrize("interval,decays", [(0, False), (7, True), (64, False), (1000, True)])
def test_the_group_form_matches_the_oracle_and_is_the_one_that_ran(H_, interval, decays):
    """Chunks around the group size and up to nine groups, none so long that the wave is left to the two passes: outputs and
    states against the oracle, and states whose last bits are not those of the two passes."""
    lens, prefix = [0, 17, 130, 144, 100, 128], [5, 16, 31, 0, 4097, 63]
    w = W.kda_workload("group form", 80 + H_, lens, H_, prefix, resume=[True, False, True, False, True, True], snap_interval=interval)
    t = w.tensors()
    if decays:
        rng = np.random.default_rng(H_)
        a = t["alpha"].numpy()
        for val, count in ((0.0, 6), (1e-9, 6), (1e-30, 4), (0.2, 200)):
            a[rng.integers(0, a.shape[0], count), rng.integers(0, H_, count), rng.integers(0, 128, count)] = val
    got_o, got_pool, status = _gpu(w, t)
    _, two_passes, _ = _gpu(w, t, layout=3)
    assert status == 0 and not np.array_equal(got_pool, two_passes)
    heads = [0, H_ - 1]
    ref_o, ref_pool = _oracle(w, t, heads=heads)
    _close_out(got_o[:, heads], ref_o, "outputs")
    _close_state(got_pool[:, heads], ref_pool, "state pool")


@pytest.mark.parametrize("H_", [9, 17, 33])                             # CTAs of 32, 64 and 128 columns
@pytest.mark.parametrize("lens,two_passes", [([192] * 4, False), ([1500, 64, 64, 64], True), ([64, 64, 64, 1500], True), ([2000, 0, 0, 0], True)])
def test_a_wave_of_one_long_chunk_is_left_to_the_two_passes(H_, lens, two_passes):
    """The library's choice sees the lengths on the device: a wave much longer than its mean takes the form whose chain is
    the faster one per token (the same bits as when it is asked for), equal chunks take the groups (other bits)."""
    w = W.kda_workload("unequal", 41, lens, H_, [0, 100, 64, 7], snap_interval=100)
    t = w.tensors()
    got_o, got_pool, status = _gpu(w, t)
    ref_o, ref_pool, _ = _gpu(w, t, layout=3)
    assert status == 0
    assert np.array_equal(got_pool, ref_pool) == two_passes
    assert np.array_equal(got_o, ref_o) or not two_passes
    _close_state(got_pool, ref_pool, "state pool")


@pytest.mark.parametrize("H_", [9, 17, 33])                             # CTAs of 32, 64 and 128 columns
def test_the_group_form_is_bit_identical_when_chunks_are_cut_at_a_multiple_of_sixteen(H_):
    """256 tokens a request in one call, and 112 and then 144: both take the groups in CTAs of the same width, and groups are
    blocks of absolute positions, so outputs and states have the same bits."""
    whole = W.kda_workload("whole", 37, [256] * 4, H_, [0, 16, 64, 160])
    t = whole.tensors()
    want_o, want_pool, status = _gpu(whole, t)
    assert status == 0 and not np.array_equal(_gpu(whole, t, layout=3)[1], want_pool)
    pool, got_o = t["state_pool"], np.zeros_like(want_o)
    for lo, hi, s_in in ((0, 112, whole.state_in), (112, 256, whole.state_out)):
        rows = np.concatenate([np.arange(r + lo, r + hi) for r in whole.row_offsets[:-1]])
        part = W.kda_workload("part", 37, [hi - lo] * 4, H_, [int(x) + lo for x in whole.prefix_lens])
        part.num_slots = whole.num_slots
        o, pool_, status = _gpu(part, {k: (v[rows].contiguous() if k != "state_pool" else pool) for k, v in t.items()},
                                state_in=s_in, state_out=whole.state_out)
        assert status == 0
        got_o[rows], pool = o, torch.from_numpy(pool_).float()
    assert np.array_equal(got_o, want_o) and np.array_equal(pool.double().numpy(), want_pool)


def _cut(w, pieces):
    """Asserts that the library cuts this wave's chains into so many pieces (on 148 SMs, as all tests of this file assume)."""
    form, k, longest = choice(len(w.chunk_lens), int(w.num_heads), int(w.total_tokens), torch.cuda.get_device_properties(0).multi_processor_count)
    assert (form, k) == (1, pieces) and w.chunk_lens.max() <= longest, (form, k, longest)


@pytest.mark.parametrize("lens,prefix,interval", [
    ([500, 0, 480, 300, 510], [5, 3, 0, 31, 64], 0),
    ([500, 1, 480, 300, 510], [100, 7, 15, 0, 1000], 100),      # snapshots inside the pieces; a chunk of fewer blocks than pieces
])
def test_chains_cut_into_pieces_match_the_oracle(lens, prefix, interval):
    """160 chains on 148 SMs in three pieces each, whose states pass through the workspace (a sample of the heads against the
    oracle; every head against the two passes)."""
    w = W.kda_workload("pieces", 19, lens, 32, prefix, snap_interval=interval)
    _cut(w, 3)
    t = w.tensors()
    heads = [0, 13, 31]
    ref_o, ref_pool = _oracle(w, t, heads)
    got_o, got_pool, status = _gpu(w, t)
    assert status == 0
    _close_out(got_o[:, heads], ref_o, "outputs")
    _close_state(got_pool[:, heads], ref_pool, "state pool")
    two_o, two_pool, status = _gpu(w, t, layout=3)
    assert status == 0
    _close_state(got_pool, two_pool, "state pool of all heads")
    assert not np.array_equal(got_pool, two_pool)
    again_o, again_pool, _ = _gpu(w, t)
    assert np.array_equal(got_o, again_o) and np.array_equal(got_pool, again_pool)


@pytest.mark.parametrize("lens,H_,pieces,step", [
    ([256, 250, 240, 256, 251], 32, 2, 128), ([384, 330, 400, 369, 390], 32, 3, 144), ([640, 600, 633, 655, 580], 32, 4, 176),
    ([992, 976, 987], 50, 5, 176), ([1500, 1479, 1488], 50, 6, 176),
])
def test_cut_chains_have_the_bits_of_whole_ones(lens, H_, pieces, step):
    """A wave whose chains are cut against the same tokens in calls of up to `step` tokens a request, which the library does not
    cut and gives to CTAs of the same width: groups are blocks of 16 absolute positions, so outputs and states have the same
    bits."""
    w = W.kda_workload("cut", 61 + pieces, lens, H_, [16 * i for i in range(len(lens))])
    _cut(w, pieces)
    t = w.tensors()
    want_o, want_pool, status = _gpu(w, t)
    assert status == 0
    pool, got_o, done = t["state_pool"], np.zeros_like(want_o), 0
    while done < max(lens):
        part_lens = [min(step, n - done) for n in lens]
        rows = np.concatenate([np.arange(r + done, r + done + n) for r, n in zip(w.row_offsets[:-1], part_lens)])
        part = W.kda_workload("part", 61 + pieces, part_lens, H_, [int(x) + done for x in w.prefix_lens])
        part.num_slots = w.num_slots
        _cut(part, 1)
        o, pool_, status = _gpu(part, {k: (v[rows].contiguous() if k != "state_pool" else pool) for k, v in t.items()},
                                state_in=w.state_in if done == 0 else w.state_out, state_out=w.state_out)
        assert status == 0
        got_o[rows], pool = o, torch.from_numpy(pool_).float()
        done += step
    assert np.array_equal(got_o, want_o) and np.array_equal(pool.double().numpy(), want_pool)


@pytest.mark.parametrize("lens,interval", [([640, 0, 33, 600, 640], 0), ([33, 640, 0, 640, 600], 100)])
def test_a_cut_wave_that_is_turned_away_on_the_device_is_the_two_passes(lens, interval):
    """The host would cut the chains in three; the CTAs find a chunk longer than the choice allows and leave the wave, whichever
    piece they would have been, to the two passes behind: their bits."""
    w = W.kda_workload("turned away", 43, lens, 32, [5, 3, 0, 31, 64], snap_interval=interval)
    form, pieces, longest = choice(5, 32, w.total_tokens)
    assert (form, pieces) == (1, 3) and max(lens) > longest
    t = w.tensors()
    got_o, got_pool, status = _gpu(w, t)
    two_o, two_pool, two_status = _gpu(w, t, layout=3)
    assert status == 0 and two_status == 0
    assert np.array_equal(got_o, two_o) and np.array_equal(got_pool, two_pool)


@pytest.mark.parametrize("same_slot", [False, True])         # periodic snapshots in slots of their own, or in the chunk end's
def test_cut_chains_with_states_in_place_strong_decays_and_snapshots(same_slot):
    """The first piece reads the slot that the last one writes, snapshots are stored by the piece that passes them, decays end
    groups or go to the state directly (a sample of the heads against the oracle)."""
    lens, heads = [500, 0, 480, 300, 510], [0, 21, 31]
    w = W.kda_workload("in place", 67, lens, 32, [5, 3, 16, 31, 64], snap_interval=100)
    _cut(w, 3)
    w.state_in = w.state_out
    if same_slot:
        w.snap_slots[:] = w.state_out[:, None]
    t = w.tensors()
    rng, a = np.random.default_rng(3), t["alpha"].numpy()
    for val, count in ((0.0, 6), (1e-9, 6), (1e-30, 4), (0.2, 200)):
        a[rng.integers(0, a.shape[0], count), rng.choice(heads, count), rng.integers(0, 128, count)] = val
    ref_o, ref_pool = _oracle(w, t, heads)
    for _ in range(5):
        got_o, got_pool, status = _gpu(w, t)
        assert status == 0
        _close_out(got_o[:, heads], ref_o, "outputs")
        _close_state(got_pool[:, heads], ref_pool, "state pool")


def test_a_captured_call_of_cut_chains_replays_with_the_same_bits():
    """The clearing of the counter and of the hand-over flags is part of the graph: every replay starts from the first piece."""
    w = W.kda_workload("captured", 71, [500, 30, 480, 300, 510], 32, [5, 3, 0, 31, 64])
    _cut(w, 3)
    t = w.tensors()
    want_o, want_pool, status = _gpu(w, t)
    assert status == 0
    dev = torch.device("cuda")
    d = {k: v.to(dev) for k, v in t.items()}
    i32 = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).to(dev)
    rows, s_in, s_out, prefix = torch.from_numpy(w.row_offsets).to(dev), i32(w.state_in), i32(w.state_out), i32(w.prefix_lens)
    ws = torch.empty(wpp.wpp_kda_workspace_bytes(5, 32, w.total_tokens), dtype=torch.uint8, device=dev)
    status, out, pool = torch.zeros(1, dtype=torch.int32, device=dev), torch.empty_like(d["v"]), d["state_pool"].clone()
    call = lambda: wpp.wpp_kda_chunk(H.ctx(), d["q"], d["k"], d["v"], d["alpha"], d["beta"], rows, pool, s_in, s_out, out=out,
                                     prefix_lens=prefix, status=status, workspace=ws)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            call()
    for _ in range(3):
        pool.copy_(d["state_pool"])
        out.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert np.array_equal(out.float().cpu().double().numpy(), want_o)
        assert np.array_equal(pool.cpu().double().numpy(), want_pool)
