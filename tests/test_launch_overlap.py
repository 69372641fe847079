"""Kernels that let the next one in their stream be set up while they run (griddepcontrol): what the sources have to keep."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc")


def _kernels():
    """(file, kernel name, body up to the next kernel) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        starts = [m.start() for m in re.finditer(r"__global__", src)] + [len(src)]
        for a, b in zip(starts, starts[1:]):
            name = re.search(r"(\w+)\s*\(\s*const", src[a:b])
            yield os.path.basename(path), name.group(1) if name else "?", src[a:b]


def test_tensor_memory_is_allocated_before_the_next_kernel_is_let_in():
    """The next kernel may take tensor memory of the SM and keep it until this one has ended; an allocation that comes after
    the release could wait for it for ever.  Every CTA has to have passed the barrier behind its own allocation first."""
    seen = 0
    for path, name, body in _kernels():
        if "tmem_alloc(" not in body or "grid_launch_dependents()" not in body:
            continue
        seen += 1
        alloc, release = body.index("tmem_alloc("), body.index("grid_launch_dependents()")
        assert alloc < release, f"{path}: {name} lets the next kernel in before it has its tensor memory"
        assert "__syncthreads()" in body[alloc:release], f"{path}: {name} releases before all of the CTA has its tensor memory"
    assert seen >= 3


def test_an_append_grid_that_is_set_up_early_fits_the_sms():
    """What counts as such a grid is what the launch bounds make room for, whatever registers the kernel would like."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wpp_append_combine.cu")).read())
    assert re.search(r"__launch_bounds__\(256, kVec == 1 \? kAppendCtas : [^)]*\) wpp_append_kernel", src)
    assert re.search(r"q\.few = total <= \(int64_t\)num_sms \* wpp::kAppendCtas \* 256;", src)


@pytest.mark.gpu
def test_small_attention_directly_behind_the_two_pass_recurrent_layer():
    """The chain kernel takes all 512 columns of an SM's tensor memory, the small attention shape 256 per CTA: queued behind
    one another without anything between, both end with the results they have apart."""
    import numpy as np
    import torch

    import paper_2609_35263_b200 as wpp
    import wpp_workloads as W
    from tests import gpu_harness as H
    from tests.test_gpu_kda import _gpu

    w = W.custom_workload([300, 64, 0, 17], [33, 64, 90, 5], 8, 2, 64, 16, seed=23)
    g = H.device_inputs(w)
    apart = H.run_wave(w, g, shape=2)
    assert apart["status"] == 0
    kw = W.kda_workload("front", 29, [200, 70, 333], 7, [5, 0, 64])
    t = kw.tensors()
    o_apart, pool_apart, status = _gpu(kw, t, layout=3)
    assert status == 0
    dev = torch.device("cuda")
    d = {k: v.to(dev) for k, v in t.items()}
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)
    rows, s_in, s_out, prefix, chunks, P, bt = (torch.from_numpy(kw.row_offsets).to(dev), i32(kw.state_in), i32(kw.state_out),
                                                i32(kw.prefix_lens), i32(w.chunk_lens), i32(w.prefix_lens), i32(w.block_tables))
    ws = torch.empty(wpp.wpp_kda_workspace_bytes(3, 7, int(t["q"].shape[0])), dtype=torch.uint8, device=dev)
    plan, status = apart["plan"], torch.zeros(1, dtype=torch.int32, device=dev)
    ws_attn = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device=dev)
    pool0 = d["state_pool"].clone()
    for _ in range(20):
        out, out_kda = torch.zeros_like(apart["out"]), torch.zeros_like(d["v"])
        d["state_pool"].copy_(pool0)
        torch.cuda.synchronize()
        wpp.wpp_kda_chunk(H.ctx(), d["q"], d["k"], d["v"], d["alpha"], d["beta"], rows, d["state_pool"], s_in, s_out, out=out_kda,
                          prefix_lens=prefix, status=status, layout=3, workspace=ws)
        wpp.wpp_prefill_attention_varlen(H.ctx(), H.desc_of(w), g["q"], out, None, g["k_pool"], g["v_pool"], bt, P, chunks, plan,
                                         workspace=ws_attn, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert torch.equal(out, apart["out"])
        assert np.array_equal(out_kda.float().cpu().double().numpy(), o_apart)
        assert np.array_equal(d["state_pool"].cpu().double().numpy(), pool_apart)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("P,C", [([300, 64], [33, 90]), ([0, 70, 5], [700, 600, 130]), ([5000], [40])])
def test_passes_one_behind_the_other_see_their_own_keys(P, C, shape):
    """Append and attention of successive passes are set up while the kernel before them runs, append over the same pages each
    time: every pass has the results it has alone.  (Waves of one tile per CTA, of several, and cut along the keys.)"""
    import torch

    import paper_2609_35263_b200 as wpp
    import wpp_workloads as W
    from tests import gpu_harness as H

    w = W.custom_workload(P, C, 8, 2, 128, 64, seed=31, spare_pages=4)
    g, d, dev = H.device_inputs(w), H.desc_of(w), torch.device("cuda")
    plan = wpp.wpp_plan_tiles(H.ctx(), d, w.prefix_lens, w.chunk_lens, opts=wpp.PlanOpts(0, 0, 0, 0, 0, shape)).to_device(dev)
    i32 = lambda a: torch.from_numpy(a.astype("int32")).to(dev)
    Pd, Cd, bt = i32(w.prefix_lens), i32(w.chunk_lens), i32(w.block_tables)
    ws = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    new = [(g["k_new"] * f, g["v_new"] * f) for f in (1.0, -0.5, 0.25, 2.0)]

    def one(k, v, out):
        wpp.wpp_kv_append(H.ctx(), d, k, v, g["k_pool"], g["v_pool"], bt, Pd, Cd, plan, status=status)
        wpp.wpp_prefill_attention_varlen(H.ctx(), d, g["q"], out, None, g["k_pool"], g["v_pool"], bt, Pd, Cd, plan, workspace=ws, status=status)

    alone = []
    for k, v in new:
        out = torch.zeros_like(g["q"])
        one(k, v, out)
        torch.cuda.synchronize()
        alone.append(out)
    for _ in range(5):
        outs = [torch.zeros_like(g["q"]) for _ in new]
        torch.cuda.synchronize()
        for (k, v), out in zip(new, outs):
            one(k, v, out)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and all(torch.equal(a, b) for a, b in zip(alone, outs))
    assert not torch.equal(alone[0], alone[1])


@pytest.mark.gpu
@pytest.mark.parametrize("with_append", [False, True])
@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("lens,layout", [([200, 70, 333], 3), ([4096], 3), ([200], 0), ([100, 130, 64], 0)])
def test_append_and_attention_directly_behind_the_recurrent_layer(lens, layout, shape, with_append):
    """Both are set up while the kernel before them runs: behind the two passes (one segment and several; the chain kernel and the
    SM-wide attention kernel take all 512 columns of an SM's tensor memory), behind the group form alone and behind the empty two
    passes that follow it.  Every result is what it is apart."""
    import numpy as np
    import torch

    import paper_2609_35263_b200 as wpp
    import wpp_workloads as W
    from tests import gpu_harness as H
    from tests.test_gpu_kda import _gpu
    from tests.test_kda_pieces import choice
    from tests.test_kda_segments import cut

    heads = 32 if lens == [4096] else 7
    if layout == 0:
        assert choice(len(lens), heads, sum(lens))[0] > 0
    else:
        assert len(cut(len(lens), heads, sum(lens))) == (3 if lens == [4096] else 1)
    dev = torch.device("cuda")
    w = W.custom_workload([300, 64, 0, 17], [33, 64, 90, 5], 8, 2, 64, 16, seed=23)
    g = H.device_inputs(w)
    pools = g["k_pool"].clone(), g["v_pool"].clone()
    apart = H.run_wave(w, g, shape=shape)
    after = g["k_pool"].clone(), g["v_pool"].clone()
    kw = W.kda_workload("front", 29, lens, heads, [5, 0, 64][:len(lens)])
    t = kw.tensors()
    o_apart, pool_apart, status = _gpu(kw, t, layout=layout)
    assert status == 0 and apart["status"] == 0
    d = {k: v.to(dev) for k, v in t.items()}
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)
    rows, s_in, s_out, prefix = torch.from_numpy(kw.row_offsets).to(dev), i32(kw.state_in), i32(kw.state_out), i32(kw.prefix_lens)
    chunks, P, bt = i32(w.chunk_lens), i32(w.prefix_lens), i32(w.block_tables)
    ws = torch.empty(wpp.wpp_kda_workspace_bytes(len(lens), heads, sum(lens)), dtype=torch.uint8, device=dev)
    plan, status = apart["plan"], torch.zeros(1, dtype=torch.int32, device=dev)
    ws_attn = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device=dev)
    pool0 = d["state_pool"].clone()
    for _ in range(10):
        out, out_kda = torch.zeros_like(apart["out"]), torch.zeros_like(d["v"])
        d["state_pool"].copy_(pool0)
        for name, before, now in zip(("k_pool", "v_pool"), pools, after):
            g[name].copy_(before if with_append else now)
        torch.cuda.synchronize()
        for _ in range(2):                                          # (the recurrent layer behind the attention kernel as well)
            d["state_pool"].copy_(pool0)
            wpp.wpp_kda_chunk(H.ctx(), d["q"], d["k"], d["v"], d["alpha"], d["beta"], rows, d["state_pool"], s_in, s_out, out=out_kda,
                              prefix_lens=prefix, status=status, layout=layout, workspace=ws)
            if with_append:
                wpp.wpp_kv_append(H.ctx(), H.desc_of(w), g["k_new"], g["v_new"], g["k_pool"], g["v_pool"], bt, P, chunks, plan, status=status)
            wpp.wpp_prefill_attention_varlen(H.ctx(), H.desc_of(w), g["q"], out, None, g["k_pool"], g["v_pool"], bt, P, chunks, plan,
                                             workspace=ws_attn, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert torch.equal(out, apart["out"]) and torch.equal(g["k_pool"], after[0]) and torch.equal(g["v_pool"], after[1])
        assert np.array_equal(out_kda.float().cpu().double().numpy(), o_apart)
        assert np.array_equal(d["state_pool"].cpu().double().numpy(), pool_apart)
