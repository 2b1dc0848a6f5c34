"""Workloads of the eviction step (Section 4.3, Eq. 4) for timing and for comparing two builds.

A case is one call a serving or analysis program makes: the geometry of the cache, the window, the
budget and the options, and which public entry point takes it. ``prepare`` makes what such a program
has in hand before the call (cache, window queries, output buffers, workspace), ``run`` is the call.

Inputs. Keys, values and queries are N(0,1) in bf16 with three outlier channels per KV head (x4), as
in the synthetic workloads of ``synth.py``. A fourth channel carries the salience of a key: it is
large on passages (spans of neighbouring positions, at random places) and zero elsewhere, and every
window query is large there too, so the passages get the attention mass, as retrieved passages of a
long prompt do. The passages of a unit, widened by half a pooling kernel, hold exactly as many
positions as the budget selects. Pooled scores on either side of the budget then differ by far more
than rounding, the kept set does not depend on the order of a sum, and kept rows compare bit by bit.
"""
import math

import torch

from paper_2505_20334_b200 import binding as laq

_BASE = {"call": "laq_evict", "n_layers": 32, "batch": 1, "n_q_heads": 32, "n_kv_heads": 8, "head_dim": 128,
         "prompt_len": 4096, "shortest": 0, "window_len": 16, "keep_tail": 16, "local_window": 0,
         "pool_kernel": 7, "pool_mode": 0, "score_mode": 0, "group_mode": 0, "budget": 512,
         "position_major": False}


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if "keep_tail" not in kw:
        c["keep_tail"] = c["window_len"]
    if name is not None:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # one layer, one KV head, a short prompt: what a latency-bound caller pays per call
        _case("one unit, 1k", n_layers=1, n_q_heads=4, n_kv_heads=1, prompt_len=1024, window_len=8, budget=128),
        # one 4k prompt through an 8B-class model, by the convenience call that allocates its outputs
        _case("8B, 4k prompt", call="evict", prompt_len=4096, budget=512),
        # a serving batch: prompts of different (odd) lengths in a position-major cache, LAQ++ window
        _case("8B, ragged batch, LAQ++", n_layers=16, batch=4, prompt_len=12001, shortest=2311, window_len=32,
              local_window=16, budget=777, position_major=True),
        # long-context batch, the headline workload of the benchmark
        _case("8B, 4 x 32k", batch=4, prompt_len=32768, window_len=32, budget=2048),
        # larger batch of mid-length prompts, smaller window
        _case("7B, 8 x 16k", batch=8, prompt_len=16384, window_len=16, pool_kernel=5, budget=512),
        # 70B-class model (eight query heads per KV head): 256 window rows per unit
        _case("70B, 64k prompt", n_layers=80, n_q_heads=64, prompt_len=65536, window_len=32, budget=2048),
        # analysis of a short lookahead (two steps): scores, selection and its recall against a known set
        _case("two lookahead steps, recall", call="score_select_recall", batch=1, prompt_len=32768, window_len=2,
              keep_tail=32, budget=1024),
        # Eq. 4 read literally: raw logit sums, one pass over the keys
        _case("raw logits, 2 x 32k", batch=2, prompt_len=32768, window_len=32, score_mode=1, budget=1024),
        # every query head keeps its own set, maximum pooling
        _case("per query head, 8k", prompt_len=8192, window_len=32, group_mode=2, pool_mode=1, pool_kernel=5,
              budget=512),
        # a pyramid of per-layer budgets, odd prompt length, one ragged output pool
        _case("pyramid budgets, 6k", call="layers", prompt_len=6007, window_len=16, budget=1024),
        # a small model with 64-dim heads
        _case("64-dim heads, 4k", n_layers=16, head_dim=64, prompt_len=4096, window_len=8, budget=256),
        # a cache that was offloaded to pinned host memory: copies in, copies out
        _case("host cache, 8k", call="host", n_layers=8, prompt_len=8192, window_len=16, budget=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("small", "evict", "ragged", "long", "short window", "wide", "raw", "heads", "layers",
                       "head_dim", "host"))
    kv = rng.choice((1, 2, 4, 8))
    g = rng.choice((1, 2, 4, 8))
    w = rng.choice((4, 5, 8, 12, 16, 24, 32))
    c = {"n_layers": rng.choice((4, 8, 16, 28, 32)), "n_kv_heads": kv, "pool_kernel": rng.choice((1, 3, 5, 7, 7, 9)),
         "pool_mode": int(rng.random() < 0.25), "prompt_len": _log_int(rng, 1500, 16000)}
    if kind == "small":
        c.update(n_layers=rng.choice((1, 1, 2, 4)), n_kv_heads=rng.choice((1, 2)), prompt_len=_log_int(rng, 300, 4000))
    elif kind == "evict":
        c.update(call="evict", batch=rng.choice((1, 1, 2)))
    elif kind == "ragged":
        c.update(batch=rng.randint(2, 8), local_window=rng.randint(0, w), position_major=rng.random() < 0.5)
    elif kind == "long":
        c.update(n_layers=rng.choice((16, 32)), n_kv_heads=8, batch=rng.choice((1, 2, 4)),
                 prompt_len=_log_int(rng, 16000, 65536))
        g = 4
    elif kind == "short window":
        w = rng.choice((1, 2, 4, 8))
        c.update(call=rng.choice(("laq_evict", "score_select_recall")), prompt_len=_log_int(rng, 4000, 50000))
    elif kind == "wide":
        g, w = 8, rng.choice((20, 24, 32))
        c.update(n_layers=rng.choice((20, 40, 80)), n_kv_heads=8, prompt_len=_log_int(rng, 4000, 65536))
    elif kind == "raw":
        w = rng.choice((8, 16, 32))
        c.update(score_mode=1, pool_mode=0, batch=rng.choice((1, 2)), prompt_len=_log_int(rng, 2000, 50000))
    elif kind == "heads":
        g, w = rng.choice((2, 4, 8)), rng.choice((8, 16, 32))
        c.update(group_mode=rng.choice((1, 2)))
    elif kind == "layers":
        c.update(call="layers")
    elif kind == "head_dim":
        d = rng.choice((64, 64, 80, 96, 256))
        w = rng.choice((4, 8, 16))
        c.update(head_dim=d, n_layers=rng.choice((2, 4, 8)), prompt_len=_log_int(rng, 500, 6000))
    else:
        c.update(call="host", n_layers=rng.choice((1, 2, 4)), n_kv_heads=rng.choice((1, 8)))
    length = c["prompt_len"]
    k = c["pool_kernel"]
    # budgets of the configurations (128 .. 2048), at most a quarter of the shortest prompt
    shortest = max(300, length // rng.randint(2, 6)) if kind == "ragged" else 0
    most = (shortest or length) // 4
    budget = min(_log_int(rng, 100, 2100), most)
    budget = max(budget, w + 2 * k)
    case = _case(window_len=w, n_q_heads=c["n_kv_heads"] * g, budget=budget, shortest=shortest, **c)
    # never more than the largest listed case: 2^30 x 10 window-row-key pairs, 8 GiB of keys
    while case["n_layers"] > 1 and (_pairs(case) > 1.0e10 or _key_bytes(case) > 8.0e9 or
                                    (case["head_dim"] != 128 and _pairs(case) > 6.0e7) or
                                    (case["call"] == "host" and _key_bytes(case) > 1.5e8)):
        case["n_layers"] = (case["n_layers"] + 1) // 2
    return case


# ------------------------------------------------------------------------------- sizes of a case
def _lens(c):
    """Prompt lengths of the batch: the allocated length, or spread from it down to `shortest`."""
    if not c["shortest"]:
        return [c["prompt_len"]] * c["batch"]
    step = (c["prompt_len"] - c["shortest"]) / max(1, c["batch"] - 1)
    return [int(c["prompt_len"] - step * b) for b in range(c["batch"])]


def _budgets(c):
    """Budgets of the layers: one for all, or falling from `budget` to a quarter of it (layers call)."""
    n = c["n_layers"]
    if c["call"] != "layers":
        return [c["budget"]] * n
    least = max(c["budget"] // 4, c["keep_tail"] + 2 * c["pool_kernel"])
    return [max(least, c["budget"] - (c["budget"] - least) * i // max(1, n - 1)) for i in range(n)]


def _rows(c):
    return c["n_q_heads"] // c["n_kv_heads"] * c["window_len"]


def _pairs(c):
    return float(c["n_layers"] * c["n_kv_heads"]) * _rows(c) * sum(_lens(c))


def _key_bytes(c):
    return 2.0 * c["n_layers"] * c["n_kv_heads"] * c["head_dim"] * sum(_lens(c))


def work(case):
    """K and Q read once, the kept V rows read, the kept rows of K and V and their positions written;
    one dot product per window row and key (in raw-logit mode one per key)."""
    c = case
    row = 2.0 * c["head_dim"]
    heads = c["n_q_heads"] if c["group_mode"] == 2 else c["n_kv_heads"]
    kept = float(sum(_budgets(c))) * c["batch"] * heads
    n = _key_bytes(c) + row * c["n_layers"] * c["batch"] * c["n_q_heads"] * c["window_len"]
    flops = 2.0 * c["head_dim"] * _pairs(c)
    if c["score_mode"] == 1:
        flops /= _rows(c)
    if c["call"] == "score_select_recall":
        # scores and positions written, the known set read, one recall and one count per unit
        units = c["n_layers"] * c["batch"] * c["n_kv_heads"]
        n += 4.0 * units * (c["prompt_len"] - c["keep_tail"]) + 8.0 * kept + 8.0 * units
    else:
        n += kept * (3.0 * row + 4.0)
    return {"bytes": n, "flops": flops}


def tolerance(case):
    # kept rows and positions are exact (see the head of the file); scores are fp32 sums
    if case["call"] == "score_select_recall":
        return {"rel": 1e-5, "max": 1e-4}
    return "exact"


# ------------------------------------------------------------------------------------- inputs
def _passages(gen, c, budget, dev):
    """0/1 per (prompt, KV head, position): passages that, widened by half a pooling kernel on either
    side, cover budget - keep_tail positions of every unit. One passage per equal cell of the prompt."""
    h, kb = c["pool_kernel"] // 2, budget - c["keep_tail"]
    shape = (c["batch"], c["n_kv_heads"])
    wide = max(2 * h + 1, min(16 + 2 * h, kb))        # a widened passage of about 16 positions
    n = max(1, kb // wide)
    size = torch.full((n,), kb // n, device=dev)
    size[:kb % n] += 1
    order = torch.rand(shape + (n,), generator=gen, device=dev).argsort(dim=-1)
    size = size[order]                                # widened lengths in random order, same sum
    scored = torch.tensor([x - c["keep_tail"] for x in _lens(c)], device=dev).view(-1, 1, 1)
    cell = scored // n
    begin = torch.arange(n, device=dev) * cell + (
        torch.rand(shape + (n,), generator=gen, device=dev) * (cell - size + 1)).long()
    mark = torch.zeros(shape + (c["prompt_len"] + 1,), dtype=torch.int32, device=dev)
    one = torch.ones_like(begin, dtype=torch.int32)
    mark.scatter_add_(-1, begin + h, one)
    mark.scatter_add_(-1, begin + size - h, -one)
    return mark.cumsum(dim=-1)[..., :-1]


def _inputs(c, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(1000003 * int(seed) + 17)
    nl, bt, hq, hkv, d, length = (c[x] for x in ("n_layers", "batch", "n_q_heads", "n_kv_heads", "head_dim",
                                                 "prompt_len"))
    q = torch.randn((nl, bt, hq, c["window_len"], d), generator=gen, device=dev, dtype=torch.bfloat16)
    if c["position_major"]:                           # [.., position, head, dim] in memory
        k, v = (torch.randn((nl, bt, length, hkv, d), generator=gen, device=dev, dtype=torch.bfloat16)
                .permute(0, 1, 3, 2, 4) for _ in range(2))
    else:
        k, v = (torch.randn((nl, bt, hkv, length, d), generator=gen, device=dev, dtype=torch.bfloat16)
                for _ in range(2))
    for n, budget in enumerate(_budgets(c)):
        channels = torch.rand((hkv, d), generator=gen, device=dev).argsort(dim=-1)
        gain = torch.ones((hkv, d), device=dev).scatter_(1, channels[:, 1:4], 4.0)
        k[n] *= gain.to(torch.bfloat16).view(1, hkv, 1, d)
        # mean logit of a passage key: 14, one salience channel per KV head
        root = math.sqrt(14.0 * math.sqrt(d))
        ch = channels[:, 0].view(1, hkv, 1, 1)
        passages = _passages(gen, c, budget, dev)
        k[n].scatter_(-1, ch.expand(bt, hkv, length, 1), (root * passages).to(torch.bfloat16).unsqueeze(-1))
        qc = ch.repeat_interleave(hq // hkv, dim=1).expand(bt, hq, c["window_len"], 1)
        q[n].scatter_(-1, qc, root)
    return q, k, v


def prepare(case, seed):
    c = case
    q, k, v = _inputs(c, seed)
    nl, bt, hkv, d = c["n_layers"], c["batch"], c["n_kv_heads"], c["head_dim"]
    state = {"case": c, "lens": _lens(c) if c["shortest"] else None}
    if c["call"] == "host":
        state["q"], state["k"], state["v"] = (t.cpu().pin_memory() for t in (q, k, v))
        state["evictor"] = laq.HostEvictor(tuple(q.shape), tuple(k.shape), c["budget"], c["pool_kernel"], c["keep_tail"])
        return state
    state.update(q=q, k=k, v=v)
    if c["call"] == "evict":
        return state
    budgets = _budgets(c)
    p = laq.params_for(q, k, c["keep_tail"], c["pool_kernel"], max(budgets), v=v)
    p.local_window, p.pool_mode, p.score_mode, p.group_mode = (
        c["local_window"], c["pool_mode"], c["score_mode"], c["group_mode"])
    p.set_seq_lens(state["lens"])
    heads = c["n_q_heads"] if c["group_mode"] == laq.LAQ_GROUP_PER_HEAD else hkv
    if c["call"] == "layers":
        entries = laq.laq_layers_pool_entries(p, budgets)
        state["idx"] = torch.empty(entries, dtype=torch.int32, device=k.device)
        out = (entries, d)
        state["budgets"] = budgets
    else:
        out = (nl, bt, heads, c["budget"], d)
        state["idx"] = torch.empty(out[:-1], dtype=torch.int32, device=k.device)
    if c["call"] == "score_select_recall":
        state["scores"] = torch.empty((nl, bt, heads, c["prompt_len"] - c["keep_tail"]), dtype=torch.float32,
                                      device=k.device)
        # the known set: the same number of positions, evenly spaced over the prompt
        gold = torch.arange(c["budget"], device=k.device, dtype=torch.int64) * c["prompt_len"] // c["budget"]
        state["gold"] = gold.to(torch.int32).expand(nl, bt, heads, c["budget"]).contiguous()
    else:
        state["k_out"] = torch.empty(out, dtype=torch.bfloat16, device=k.device)
        state["v_out"] = torch.empty_like(state["k_out"])
        if c["call"] == "laq_evict":
            for i, dim in enumerate(("layer", "batch", "head", "pos")):
                setattr(p, f"o_stride_{dim}", state["k_out"].stride(i))
    state["params"], state["ws"] = p, laq.alloc_workspace(p, k.device)
    return state


def run(state):
    s, c = state, state["case"]
    if c["call"] == "evict":
        out = laq.evict(s["q"], s["k"], s["v"], c["budget"], pool_kernel=c["pool_kernel"], keep_tail=c["keep_tail"],
                        local_window=c["local_window"], pool_mode=c["pool_mode"], score_mode=c["score_mode"],
                        seq_lens=s["lens"], group_mode=c["group_mode"])
        return out["k_out"], out["v_out"], out["idx"]
    if c["call"] == "laq_evict":
        laq.laq_evict(s["params"], s["q"], s["k"], s["v"], s["k_out"], s["v_out"], s["idx"], None, s["ws"])
        return s["k_out"], s["v_out"], s["idx"]
    if c["call"] == "layers":
        laq.laq_evict_layers(s["params"], s["budgets"], s["q"], s["k"], s["v"], s["k_out"], s["v_out"], s["idx"], None,
                             s["ws"])
        return s["k_out"], s["v_out"], s["idx"]
    if c["call"] == "score_select_recall":
        laq.laq_score(s["params"], s["q"], s["k"], s["scores"], s["ws"])
        laq.laq_select(s["params"], s["scores"], s["idx"])
        recall, common = laq.laq_recall(s["idx"], s["gold"])
        return s["scores"], s["idx"], recall, common
    return s["evictor"].run(s["q"], s["k"], s["v"])
