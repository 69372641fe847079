"""KV append alone: bit-exact against the oracle over the entire pools, including odd bit patterns."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_35263_b200 as wpp
import wpp_workloads as W
from tests.helpers import bits, cpu_inputs, from_bits
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,C,Hkv,d,B", [
    ([0], [1], 1, 64, 16),
    ([37, 0, 129], [200, 1, 64], 2, 128, 16),
    ([5, 130, 257, 0], [400, 1, 127, 0], 4, 64, 32),
    ([4096], [3000], 8, 128, 64),
    ([1, 2, 3], [300, 300, 300], 2, 128, 128),
])
def test_append_is_bit_exact(P, C, Hkv, d, B):
    w = W.custom_workload(P, C, Hkv * 2, Hkv, d, B, seed=21, spare_pages=7)
    inp = cpu_inputs(w)
    kn = bits(inp["k_new"]).copy()
    if kn.size >= 4:
        kn.reshape(-1)[:4] = [0x7FC1, 0x8000, 0xFF80, 0xFFFF]      # NaN payload, -0, -inf, NaN
    inp["k_new"] = from_bits(kn)
    kp, vp = oracle.oracle_append(inp["k_new"], inp["v_new"], inp["k_pool"], inp["v_pool"], w.block_tables,
                                  w.prefix_lens, w.chunk_lens)
    res = H.run_wave(w, H.device_inputs(w, inp), do_attention=False)
    assert res["status"] == 0
    assert np.array_equal(bits(res["k_pool"]), kp)
    assert np.array_equal(bits(res["v_pool"]), vp)


@pytest.mark.parametrize("R,most,Hkv,d,B", [(33, 5, 1, 64, 16), (1100, 3, 1, 64, 16), (70, 40, 3, 128, 32), (700, 30, 5, 64, 16), (45, 170, 8, 128, 64)])
def test_append_finds_every_request(R, most, Hkv, d, B):
    """More requests than one search step tells apart, empty chunks among them, several requests' tokens in a warp, and sizes on
    both sides of the one from which a thread moves several vectors (303,104 vectors on 148 SMs; the last two)."""
    rng = np.random.default_rng(R)
    C = rng.integers(0, most + 1, R).tolist()
    C[0], C[-1] = 0, max(1, C[-1])
    w = W.custom_workload(rng.integers(0, 50, R).tolist(), C, Hkv, Hkv, d, B, seed=R, spare_pages=3)
    inp = cpu_inputs(w)
    kp, vp = oracle.oracle_append(inp["k_new"], inp["v_new"], inp["k_pool"], inp["v_pool"], w.block_tables, w.prefix_lens, w.chunk_lens)
    res = H.run_wave(w, H.device_inputs(w, inp), do_attention=False)
    assert res["status"] == 0
    assert np.array_equal(bits(res["k_pool"]), kp) and np.array_equal(bits(res["v_pool"]), vp)


def test_append_does_not_walk_over_empty_chunks():
    """The second token of a warp may belong to a request far behind that of its first one: no slower than with the next one (a
    walk from request to request over 30,000 of them takes a hundred times as long)."""
    R, dev = 30000, torch.device("cuda")
    k = torch.randn(2, 1, 64, device=dev).bfloat16()
    pool = torch.zeros(2, 1, 16, 64, dtype=torch.bfloat16, device=dev)
    d = wpp.make_desc(R, 1, 1, 64, 16, 1, 2)
    P, status, best = np.zeros(R, np.int32), torch.zeros(1, dtype=torch.int32, device=dev), {}
    for behind in (1, R - 1):
        C = np.zeros(R, np.int32)
        C[0] = C[behind] = 1
        bt = torch.zeros(R, 1, dtype=torch.int32, device=dev)
        bt[behind] = 1
        plan = wpp.wpp_plan_tiles(H.ctx(), d, P, C).to_device()
        Pd, Cd = torch.from_numpy(P).to(dev), torch.from_numpy(C).to(dev)
        for _ in range(20):
            pool.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            wpp.wpp_kv_append(H.ctx(), d, k, k, pool, pool, bt, Pd, Cd, plan, status=status)
            b.record()
            torch.cuda.synchronize()
            best[behind] = min(best.get(behind, 1e9), a.elapsed_time(b))
            assert torch.equal(pool[:, 0, 0], k[:, 0]) and int(status.item()) == 0
    assert best[R - 1] < 5 * best[1], best


@pytest.mark.parametrize("gaps", [(0, 1, 2, 3), (4, 5, 7, 8), (15, 16, 17, 31), (63, 64, 100, 333)])
def test_append_steps_over_any_number_of_empty_chunks(gaps):
    C = []
    for n in gaps + gaps:
        C += [2] + [0] * n + [1]
    for tail in (0, 1, 6):
        lens = C + [0] * tail
        w = W.custom_workload([i % 7 for i in range(len(lens))], lens, 1, 1, 64, 16, seed=len(lens), spare_pages=3)
        inp = cpu_inputs(w)
        kp, vp = oracle.oracle_append(inp["k_new"], inp["v_new"], inp["k_pool"], inp["v_pool"], w.block_tables, w.prefix_lens, w.chunk_lens)
        res = H.run_wave(w, H.device_inputs(w, inp), do_attention=False)
        assert res["status"] == 0
        assert np.array_equal(bits(res["k_pool"]), kp) and np.array_equal(bits(res["v_pool"]), vp)


def test_append_shared_prefix_pages_are_left_alone():
    rng = np.random.default_rng(22)
    w = W.make_workload("shared", 22, rng, [128, 150, 128], [64, 10, 100], 4, 2, 128, 64, shared_tokens=128,
                        sharers=[True, True, True], spare_pages=3)
    inp = cpu_inputs(w)
    kp, vp = oracle.oracle_append(inp["k_new"], inp["v_new"], inp["k_pool"], inp["v_pool"], w.block_tables,
                                  w.prefix_lens, w.chunk_lens)
    res = H.run_wave(w, H.device_inputs(w, inp), do_attention=False)
    assert np.array_equal(bits(res["k_pool"]), kp) and np.array_equal(bits(res["v_pool"]), vp)
    shared = w.block_tables[0, :2]
    assert np.array_equal(bits(res["k_pool"])[shared], bits(inp["k_pool"])[shared])
