"""The work a prefill stage has this library do, as measurable cases.

Four kinds of pass, each through the package's public calls:

  layer   KV append and chunked-prefill attention of one layer over a wave whose plan is held (a stage runs many layers
          per wave with one plan)
  wave    the same with the wave's plan made and copied to the device inside the pass (a stage's first layer of a wave)
  kda     the recurrent-state layer of a wave (workspace held, the library chooses the form)
  hash    chained block hashes of a batch of prompts (the step that finds the reusable prefix)

Ragged lengths are drawn from the case's own `lengths` number, so that the work of a case is fixed; values and physical
page ids come from the seed.
"""
import math

import numpy as np
import torch

import paper_2609_35263_b200 as wpp

_CTX = None


def _ctx():
    global _CTX
    if _CTX is None:
        _CTX = wpp.Context(torch.cuda.current_device())
    return _CTX


# ------------------------------------------------------------------------------------------------------------ cases
def _attn(name, kind, requests, chunk, prefix, heads, lengths=0, shared=0, sharers=0.0, suffix=0, lse=False, k_scale=False,
          page_rounded=False):
    """chunk, prefix: (least, most) tokens, uniform per request; heads: (query heads, KV heads, head_dim, page size);
    shared: tokens of a prefix that a share `sharers` of the requests has in common, each with up to `suffix` more."""
    c = dict(kind=kind, requests=requests, chunk_min=chunk[0], chunk_max=chunk[1], prefix_min=prefix[0], prefix_max=prefix[1],
             q_heads=heads[0], kv_heads=heads[1], head_dim=heads[2], page_size=heads[3], lengths=lengths, shared=shared,
             sharers=sharers, suffix=suffix, lse=lse, k_scale=k_scale, page_rounded=page_rounded)
    return dict(c, name=name) if name else c


def _kda(name, requests, chunk, heads, lengths=0, prefix=65536, snap_interval=0):
    c = dict(kind="kda", requests=requests, chunk_min=chunk[0], chunk_max=chunk[1], heads=heads, lengths=lengths, prefix=prefix,
             snap_interval=snap_interval)
    return dict(c, name=name) if name else c


def _hash(name, requests, tokens, block, lengths=0):
    c = dict(kind="hash", requests=requests, tokens_min=tokens[0], tokens_max=tokens[1], block=block, lengths=lengths)
    return dict(c, name=name) if name else c


_SMALL_HEADS, _MID_HEADS, _BIG_HEADS = (8, 2, 64, 16), (32, 8, 128, 64), (64, 8, 128, 64)


def listed():
    return [
        # one request alone on the stage: 128 new tokens behind 256 cached ones; host calls and launches are what counts
        _attn("single_request", "layer", 1, (128, 128), (256, 256), _SMALL_HEADS),
        # the wave a planner emits when little work is left: 32 short prompts, nothing cached
        _attn("short_prompts", "layer", 32, (64, 64), (0, 0), _BIG_HEADS),
        # prompts of a few hundred tokens and of a thousand, nothing cached
        _attn("prompts_256", "layer", 32, (256, 256), (0, 0), _BIG_HEADS),
        _attn("prompts_1024", "layer", 32, (1024, 1024), (0, 0), _BIG_HEADS),
        # follow-up turns: a short question behind a long cached conversation
        _attn("short_turns_long_prefix", "layer", 32, (64, 64), (32768, 32768), _BIG_HEADS),
        # an ordinary ragged wave with private page-rounded prefixes, planned inside the pass
        _attn("ragged_wave_16", "wave", 16, (256, 2048), (0, 8192), _MID_HEADS, lengths=2, lse=True, page_rounded=True),
        # concurrency 128, four fifths of the requests behind one shared 16,384-token prefix, planned inside the pass
        _attn("high_reuse_128", "wave", 128, (256, 4096), (0, 8192), _BIG_HEADS, lengths=3, shared=16384, sharers=0.8, suffix=4096),
        # long documents: 98,304 cached tokens, 8,192 new ones, keys whose scale changes along the sequence
        _attn("long_context", "layer", 2, (8192, 8192), (98304, 98304), _BIG_HEADS, lse=True, k_scale=True),
        # the recurrent layer of a 16,384-token wave over eight lanes, resumed from snapshots, and of one long prompt
        # with periodic snapshots
        _kda("recurrent_8x2048", 8, (2048, 2048), 32),
        _kda("recurrent_1x16384", 1, (16384, 16384), 32, snap_interval=4096),
        # the recurrent layer of a wave of chunk tails
        _kda("recurrent_tails", 32, (1, 63), 32, lengths=5),
        # block hashes of 64 long prompts
        _hash("hash_prompts", 64, (200000, 200000), 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    lengths = rng.randrange(1, 1 << 30)
    if what < 0.65:
        heads = rng.choice([_SMALL_HEADS, _MID_HEADS, _BIG_HEADS, _BIG_HEADS, (32, 8, 128, 128), (16, 4, 64, 32), (40, 8, 128, 64)])
        hi = _log_int(rng, 1, 8192)
        lo = hi if rng.random() < 0.3 else max(1, int(hi * rng.random()))
        prefix = 0 if rng.random() < 0.3 else _log_int(rng, 16, 131072)
        case = _attn(None, rng.choice(["layer", "layer", "wave"]), _log_int(rng, 1, 128), (lo, hi), (int(prefix * rng.random()), prefix),
                     heads, lengths=lengths, lse=rng.random() < 0.3, page_rounded=rng.random() < 0.3)
        if rng.random() < 0.3:
            case["shared"] = heads[3] * _log_int(rng, 1, 16384 // heads[3])
            case["sharers"] = round(rng.uniform(0.3, 1.0), 2)
            case["suffix"] = rng.randrange(0, 4097)
        # no dearer than a wave of a stage's budget: fewer requests until it is
        while case["requests"] > 1 and (work(case)["flops"] > 3e13 or work(case)["bytes"] > 8e9):
            case["requests"] = (case["requests"] + 1) // 2
        return case
    if what < 0.8:
        hi = _log_int(rng, 64, 16384)
        requests = _log_int(rng, 1, max(1, 16384 // hi))
        return _kda(None, requests, (max(1, hi // 2) if rng.random() < 0.5 else hi, hi), rng.choice([8, 16, 32]), lengths=lengths,
                    prefix=rng.randrange(0, 65537), snap_interval=rng.choice([0, 0, 256, 1024, 4096]))
    if what < 0.9:
        return _kda(None, _log_int(rng, 1, 64), (1, _log_int(rng, 1, 63)), rng.choice([8, 16, 32]), lengths=lengths,
                    prefix=rng.randrange(0, 65537))
    hi = _log_int(rng, 128, 200000)
    block = rng.choice([16, 32, 64, 128])
    return _hash(None, _log_int(rng, 1, 64), (max(block, hi // 4), hi), block, lengths=lengths)


# ----------------------------------------------------------------------------------------------------------- lengths
def _lengths(case):
    """Chunk and prefix lengths of a case's requests and which of them have the shared prefix."""
    rng = np.random.default_rng(case["lengths"])
    n, B = case["requests"], case["page_size"]
    C = rng.integers(case["chunk_min"], case["chunk_max"] + 1, n)
    P = rng.integers(case["prefix_min"], case["prefix_max"] + 1, n)
    share = rng.permutation(n) < int(round(n * case["sharers"])) if case["shared"] else np.zeros(n, bool)
    P = np.where(share, case["shared"] + rng.integers(0, case["suffix"] + 1, n), P)
    if case["page_rounded"]:
        P = P // B * B
    return C.astype(np.int64), P.astype(np.int64), share


def _span(case, least, most):
    return np.random.default_rng(case["lengths"]).integers(case[least], case[most] + 1, case["requests"]).astype(np.int64)


# ----------------------------------------------------------------------------------------------------------- attention
def _prepare_attn(case, seed):
    C, P, share = _lengths(case)
    R, B, Hq, Hkv, d = case["requests"], case["page_size"], case["q_heads"], case["kv_heads"], case["head_dim"]
    T = int(C.sum())
    # block tables: the shared pages first, then every request's own, from one permutation of the pool
    shared_blocks = case["shared"] // B if share.any() else 0
    blocks = (P + C + B - 1) // B
    own = blocks - shared_blocks * share
    pages = int(shared_blocks + own.sum()) + 16
    perm = np.random.default_rng(seed).permutation(pages).astype(np.int32)
    table = np.full((R, int(blocks.max())), -1, np.int32)
    at = shared_blocks
    for i in range(R):
        if share[i]:
            table[i, :shared_blocks] = perm[:shared_blocks]
        table[i, blocks[i] - own[i]:blocks[i]] = perm[at:at + own[i]]
        at += int(own[i])
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    bf16 = dict(dtype=torch.bfloat16, device=dev)
    s = dict(q=torch.empty(T, Hq, d, **bf16).normal_(generator=gen),
             k_new=torch.empty(T, Hkv, d, **bf16).normal_(generator=gen), v_new=torch.empty(T, Hkv, d, **bf16).normal_(generator=gen),
             k_cache=torch.empty(pages, Hkv, B, d, **bf16).normal_(generator=gen),
             v_cache=torch.empty(pages, Hkv, B, d, **bf16).normal_(generator=gen),
             out=torch.empty(T, Hq, d, **bf16))
    if case["k_scale"]:
        # keys twice as large on every other stretch of 4,096 positions
        page_scale = np.ones(pages, np.float32)
        for i in range(R):
            page_scale[table[i, :blocks[i]]] = 1 + (np.arange(blocks[i]) * B // 4096 % 2)
        new_scale = np.concatenate([1.0 + (P[i] + np.arange(C[i])) // 4096 % 2 for i in range(R)])
        s["k_cache"] *= torch.from_numpy(page_scale).to(**bf16).view(-1, 1, 1, 1)
        s["k_new"] *= torch.from_numpy(new_scale).to(**bf16).view(-1, 1, 1)
    s["lse"] = torch.empty(T, Hq, dtype=torch.float32, device=dev) if case["lse"] else None
    s["prefix"], s["chunks"] = P.astype(np.int32), C.astype(np.int32)
    s["table_dev"], s["prefix_dev"], s["chunks_dev"] = (torch.from_numpy(x).to(dev) for x in (table, s["prefix"], s["chunks"]))
    s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    s["desc"] = wpp.make_desc(R, Hq, Hkv, d, B, table.shape[1], pages)
    plan = wpp.wpp_plan_tiles(_ctx(), s["desc"], s["prefix"], s["chunks"])
    s["workspace"] = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device=dev)
    if case["kind"] == "layer":
        s["plan"] = plan.to_device(dev)
    else:
        # plans of successive waves go through a ring of pinned buffers, each reused once its copy has been made
        s["ring"] = [dict(host=torch.empty(plan.host.numel(), dtype=torch.uint8, pin_memory=True),
                          dev=torch.empty(plan.plan_bytes, dtype=torch.uint8, device=dev), copied=torch.cuda.Event()) for _ in range(4)]
        s["turn"] = 0
    return s


def _run_attn(case, s):
    ctx = _ctx()
    if case["kind"] == "layer":
        plan = s["plan"]
    else:
        slot = s["ring"][s["turn"] % len(s["ring"])]
        s["turn"] += 1
        slot["copied"].synchronize()
        plan = wpp.wpp_plan_tiles(ctx, s["desc"], s["prefix"], s["chunks"], out=slot["host"]).to_device(out=slot["dev"])
        slot["copied"].record()
    wpp.wpp_kv_append(ctx, s["desc"], s["k_new"], s["v_new"], s["k_cache"], s["v_cache"], s["table_dev"], s["prefix_dev"],
                      s["chunks_dev"], plan, status=s["status"])
    wpp.wpp_prefill_attention_varlen(ctx, s["desc"], s["q"], s["out"], s["lse"], s["k_cache"], s["v_cache"], s["table_dev"],
                                     s["prefix_dev"], s["chunks_dev"], plan, workspace=s["workspace"], status=s["status"])
    return dict(out=s["out"], lse=s["lse"], k_cache=s["k_cache"], v_cache=s["v_cache"], status=s["status"])


def _work_attn(case):
    C, P, share = _lengths(case)
    Hq, Hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    T = int(C.sum())
    cached = int(P.sum()) - (case["shared"] * max(0, int(share.sum()) - 1))      # the shared prefix is read once
    kv_row = 2 * 2 * Hkv * d
    return {"bytes": 2 * 2 * T * Hq * d + (4 * T * Hq if case["lse"] else 0) + cached * kv_row + 2 * T * kv_row,
            "flops": 4 * d * Hq * int((C * P + C * (C + 1) // 2).sum())}


# ----------------------------------------------------------------------------------------------------- recurrent layer
def _prepare_kda(case, seed):
    C = _span(case, "chunk_min", "chunk_max")
    R, H, D, T = case["requests"], case["heads"], 128, int(C.sum())
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)

    def normal(*shape):
        return torch.empty(*shape, dtype=torch.float32, device=dev).normal_(generator=gen)

    interval, snaps, slots = case["snap_interval"], None, 2 * R
    if interval:
        counts = (case["prefix"] + C) // interval - case["prefix"] // interval
        snaps = np.full((R, max(1, int(counts.max()))), -1, np.int32)
        for i in range(R):
            snaps[i, :counts[i]] = slots + np.arange(counts[i])
            slots += int(counts[i])
    s = dict(q=(normal(T, H, D) * D ** -0.5).bfloat16(), k=torch.nn.functional.normalize(normal(T, H, D), dim=-1).bfloat16(),
             v=normal(T, H, D).bfloat16(), alpha=torch.sigmoid(4 + 2 * normal(T, H, D)), beta=torch.sigmoid(normal(T, H)),
             pool=0.1 * normal(slots, H, D, D), out=torch.empty(T, H, D, dtype=torch.bfloat16, device=dev), interval=interval)
    # request i resumes from slot i and leaves its state in slot R + i; periodic snapshots go to the slots after those
    s["rows"] = torch.from_numpy(np.concatenate([[0], np.cumsum(C)]).astype(np.int64)).to(dev)
    s["state_in"] = torch.arange(R, dtype=torch.int32, device=dev)
    s["state_out"] = s["state_in"] + R
    s["prefix"] = torch.full((R,), case["prefix"], dtype=torch.int32, device=dev)
    s["snaps"] = None if snaps is None else torch.from_numpy(snaps).to(dev)
    s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    s["workspace"] = torch.empty(wpp.wpp_kda_workspace_bytes(R, H, T), dtype=torch.uint8, device=dev)
    _ctx()
    return s


def _run_kda(case, s):
    wpp.wpp_kda_chunk(_ctx(), s["q"], s["k"], s["v"], s["alpha"], s["beta"], s["rows"], s["pool"], s["state_in"], s["state_out"],
                      out=s["out"], prefix_lens=s["prefix"], snap_interval=s["interval"], snap_slots=s["snaps"], status=s["status"],
                      workspace=s["workspace"])
    return dict(out=s["out"], states=s["pool"], status=s["status"])


def _work_kda(case):
    C, H, D = _span(case, "chunk_min", "chunk_max"), case["heads"], 128
    T, interval = int(C.sum()), case["snap_interval"]
    snaps = int(((case["prefix"] + C) // interval - case["prefix"] // interval).sum()) if interval else 0
    return {"bytes": T * H * (4 * 2 * D + 4 * D + 4) + (2 * case["requests"] + snaps) * H * D * D * 4, "flops": 7 * T * H * D * D}


# --------------------------------------------------------------------------------------------------------------- hashes
def _prepare_hash(case, seed):
    n = _span(case, "tokens_min", "tokens_max")
    offsets = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    blocks = np.concatenate([[0], np.cumsum(n // case["block"])]).astype(np.int64)
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    _ctx()
    return dict(tokens=torch.randint(0, 160000, (int(offsets[-1]),), dtype=torch.int32, device=dev, generator=gen),
                offsets=torch.from_numpy(offsets).to(dev), blocks=torch.from_numpy(blocks).to(dev), total=int(blocks[-1]),
                out=torch.empty(int(blocks[-1]), dtype=torch.int64, device=dev))


def _run_hash(case, s):
    return wpp.wpp_hash_blocks(_ctx(), s["tokens"], s["offsets"], s["blocks"], case["block"], salt=7, total_blocks=s["total"], out=s["out"])


def _work_hash(case):
    n = _span(case, "tokens_min", "tokens_max")
    return {"bytes": 4 * int((n // case["block"] * case["block"]).sum()) + 8 * int((n // case["block"]).sum()) + 16 * (len(n) + 1), "flops": 0}


# ------------------------------------------------------------------------------------------------------------ interface
_KINDS = {"layer": (_prepare_attn, _run_attn, _work_attn), "wave": (_prepare_attn, _run_attn, _work_attn),
          "kda": (_prepare_kda, _run_kda, _work_kda), "hash": (_prepare_hash, _run_hash, _work_hash)}


def prepare(case, seed):
    return case, _KINDS[case["kind"]][0](case, seed)


def run(state):
    case, s = state
    return _KINDS[case["kind"]][1](case, s)


def work(case):
    return _KINDS[case["kind"]][2](case)


def tolerance(case):
    # Four times what was seen between correct ways of computing a case: attention with other tile shapes and with every
    # tile cut along the keys (2.8e-3 and 6e-2: bf16 probabilities and outputs, where a tie of the rounding moves an
    # element by a step), the recurrent layer in its other forms (1.6e-4 and 7.8e-3: bf16 outputs of fp32 states).
    if case["kind"] == "hash":
        return "exact"
    if case["kind"] == "kda":
        return {"rel": 7e-4, "max": 3.2e-2}
    return {"rel": 1.1e-2, "max": 0.24}
