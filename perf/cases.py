"""Workloads whose speed matters to a user of libams: one compression event each, through the Python binding.

A pass is what a serving loop does at an event: it refreshes the device copy of its block table and lengths and calls
`AmsCompressor.compress` (or, where it cannot allocate, `select_static`).  Geometries, budgets and windows are those of
the repository's configurations (`inputs.CONFIGS`) and tests; the rest is generic.  `draw` makes more of the same
ranges: 1 to 80 layers, 1 to 64 sequences of 1 K to 128 K tokens (equal, ragged or a little above the budget),
budgets of 64 to 8192, 1 to 512 query rows per KV head, groups of 1 to 8 query heads, every scorer.
"""
import math

import numpy as np
import torch

from paper_2605_23200_b200 import binding

DEVICE = "cuda:0"
PAGE, D = 16, 128
SCORERS = {"tova": binding.AMS_SCORER_TOVA, "keydiff": binding.AMS_SCORER_KEYDIFF,
           "external": binding.AMS_SCORER_EXTERNAL, "expected": binding.AMS_SCORER_EXPECTED}
MAX_KV_BYTES = 10 << 30      # K and V of a drawn case (the largest listed one holds 43 GB)
MAX_LOGITS = 1 << 34         # (query row, token) pairs of a drawn case (the largest listed one has 4.3e10)


def _case(name, scorer, layers, q_heads, kv_heads, batch, t_min, t_max, budget, *, window=0, cap=0, segments=10, l_max=256,
          beta=0.9, pool=1, decoupled=False, carried=False):
    """t_min..t_max: cached tokens per sequence; cap: the handle's capacity in tokens; carried: credit of earlier events."""
    c = dict(scorer=scorer, layers=layers, q_heads=q_heads, kv_heads=kv_heads, batch=batch, t_min=t_min, t_max=t_max,
             budget=budget, window=window, cap=cap or -(-t_max // PAGE) * PAGE, segments=segments, l_max=l_max, beta=beta,
             pool=pool, decoupled=decoupled, carried=carried)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest event: one layer at a time, one sequence, last-query scores; launches and latency count
        _case("one_layer_4k_w1", "tova", 1, 32, 8, 1, 4096, 4096, 1024, window=1),
        # selection for a caller that cannot allocate (a stream capture in progress): eight score rows
        _case("no_alloc_8x16k", "static", 1, 8, 8, 1, 16384, 16384, 2048),
        # an 8B-class model after a 16 K prompt, 32 observation queries
        _case("8b_16k_w32", "tova", 32, 32, 8, 1, 16384, 16384, 2048, window=32),
        # a serving batch of a 7B-class model with ragged prompts: first event
        _case("7b_b16_ragged_w1", "tova", 28, 28, 4, 16, 8192, 32768, 4096, window=1, cap=32768),
        # the same batch at each later event: 128 tokens above the budget, credit carried
        _case("7b_b16_steady_w1", "tova", 28, 28, 4, 16, 4224, 4224, 4096, window=1, cap=32768, carried=True),
        # middle-sized windows, short ragged prompts, a budget that does not fill its last page
        _case("8b_b8_short_w8", "tova", 32, 32, 8, 8, 1900, 9001, 1000, window=8),
        # key-only scores on a large batch (four of the model's layers per call), no credit
        _case("keydiff_b64_32k", "keydiff", 4, 32, 8, 64, 32768, 32768, 2048, segments=16, l_max=4096, beta=1.0),
        # the longest prompt of a 70B-class model, 64 observation queries: the largest call
        _case("70b_128k_w64", "tova", 80, 64, 8, 1, 131072, 131072, 8192, window=64, segments=32, l_max=8192),
        # its later events: 512 tokens above the budget under the same capacity
        _case("70b_steady_w64", "tova", 80, 64, 8, 1, 8704, 8704, 8192, window=64, cap=131072, segments=32, l_max=8192, carried=True),
        # expected-attention scores on the 8B geometry
        _case("8b_16k_expected", "expected", 32, 32, 8, 1, 16384, 16384, 2048),
        # window attention as the mass (smoothed), expected attention as the rank: group of 7, odd ragged lengths
        _case("7b_b4_decoupled", "expected", 28, 28, 4, 4, 5003, 12011, 2048, window=16, pool=7, decoupled=True),
        # scores from the caller's own scorer: selection and compaction alone
        _case("external_b2_8k", "external", 32, 32, 8, 2, 7001, 8191, 1000, carried=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tova", "tova", "tova", "tova", "keydiff", "expected", "decoupled", "external", "static"])
    budget = _log_int(rng, 64, 8192)
    if kind == "static":
        t = _log_int(rng, 1024, 32768)
        return _case(None, "static", 1, 8, rng.randint(1, 8), 1, t, t, min(budget, t // 2), segments=rng.choice([10, 16, 32]),
                     l_max=rng.choice([256, 512, 1024]))
    q_heads, kv_heads = rng.choice([(32, 8), (28, 4), (64, 8), (40, 8), (16, 8), (8, 8)])
    group = q_heads // kv_heads
    layers, batch = _log_int(rng, 1, 80), _log_int(rng, 1, 64)
    carried = rng.random() < 0.35
    if carried:
        t_max = max(1024, budget + rng.randint(32, 1024))
        budget = max(budget, t_max - 1024)
        cap = min(131072, t_max * rng.choice([1, 2, 8]))
    else:
        t_max = _log_int(rng, 1024, 131072)
        budget = min(budget, t_max // 2)
        cap = t_max
    t_min = t_max if batch == 1 or rng.random() < 0.3 else max(budget + 1, int(t_max * rng.uniform(0.3, 1.0)))
    window = 0
    if kind in ("tova", "decoupled"):
        window = rng.choice([1, 1, _log_int(rng, 2, 64), _log_int(rng, 8, 64)])
        window = max(1, min(window, 512 // group))
    while batch * layers > 1 and (2 * layers * batch * cap * kv_heads * D * 2 > MAX_KV_BYTES
                                  or layers * batch * q_heads * max(window, 1) * t_max > MAX_LOGITS):
        if batch >= layers:
            batch -= (batch + 3) // 4
        else:
            layers -= (layers + 3) // 4
    segments = rng.choice([10, 10, 16, 32])
    l_max = rng.choice([256, 256, 512, -(-2 * t_max // segments)])
    return _case(None, "expected" if kind == "decoupled" else kind, layers, q_heads, kv_heads, batch, t_min, t_max, budget,
                 window=window, cap=-(-cap // PAGE) * PAGE, segments=segments, l_max=l_max, beta=rng.choice([0.9, 0.9, 1.0]),
                 pool=rng.choice([1, 5, 7]) if kind == "decoupled" else 1, decoupled=kind == "decoupled", carried=carried)


def _lens(case):
    """Lengths of the batch, spread over [t_min, t_max]; part of the case, so that its work is known."""
    span = case["t_max"] - case["t_min"]
    return [case["t_min"] + int(round(span * ((b + 1) * 0.6180339887 % 1.0))) for b in range(case["batch"])]


def _config(case):
    return binding.default_config(
        n_layers=case["layers"], n_q_heads=case["q_heads"], n_kv_heads=case["kv_heads"], max_batch=case["batch"],
        max_seq_len=case["cap"], max_window=case["window"], max_budget=case["budget"], max_segments=case["segments"],
        l_max=case["l_max"], ema_beta=case["beta"], pool_kernel=case["pool"], decoupled=int(case["decoupled"]),
        expected_scorer=int(case["scorer"] == "expected"))


def _scores(shape, gen):
    """Attention-like usage: log-normal, a few heavy hitters."""
    x = torch.randn(shape, generator=gen, device=DEVICE).mul_(1.2)
    x += 3.0 * (torch.rand(shape, generator=gen, device=DEVICE) < 0.01)
    return x.exp_().mul_(1.0 / shape[-1])


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    cfg = _config(case)
    if case["scorer"] == "static":
        n, T = case["kv_heads"], case["t_max"]
        return dict(static=True, cfg=cfg, case=case, scores=_scores((n, case["cap"]), gen),
                    keep=torch.zeros((n, case["budget"]), dtype=torch.int32, device=DEVICE), T=T)
    rng = np.random.default_rng(seed)
    L, B, H, Hq, W = case["layers"], case["batch"], case["kv_heads"], case["q_heads"], case["window"]
    lens = _lens(case)
    n_dst = -(-case["budget"] // PAGE)
    n_live = sum(-(-t // PAGE) for t in lens)
    n_src = int(n_live * 1.05) + 1  # live pages lie scattered over this part of the pool, the replacement pages over the rest
    P = n_src + B * n_dst
    free = rng.permutation(n_src).astype(np.int32)
    stride = case["cap"] // PAGE
    fresh = np.full(B * stride + B, -1, np.int32)
    at = 0
    slots = []
    for b, t in enumerate(lens):
        n = -(-t // PAGE)
        pages = free[at:at + n]
        fresh[b * stride:b * stride + n] = pages
        fresh[B * stride + b] = t
        i = np.arange(t)
        slots.append(pages[i // PAGE].astype(np.int64) * PAGE + i % PAGE)
        at += n
    dst = (n_src + rng.permutation(B * n_dst)).astype(np.int32).reshape(B, n_dst)

    # keys: N(0, 1); per sequence six spans leaning towards what the queries look for, and 1 % heavy hitters; the places
    # differ from layer to layer in half of the layers at a time
    k = torch.empty((L, P, PAGE, H, D), dtype=torch.bfloat16, device=DEVICE)
    v = torch.empty_like(k)
    lean = torch.nn.functional.normalize(torch.randn((L, H, D), generator=gen, device=DEVICE), dim=-1)
    places = []
    for _ in range(2):
        spans, heavy = [], []
        for b, t in enumerate(lens):
            for i in range(0 if case["carried"] else 6):
                n = int(min(rng.integers(64, 257), t // 6))
                s = i * (t // 6) + int(rng.integers(0, t // 6 - n + 1))
                spans.append(slots[b][s:s + n])
            heavy.append(rng.choice(slots[b], size=max(1, t // 100), replace=False))
        places.append([torch.from_numpy(np.concatenate(x)).to(DEVICE) if x else None for x in (spans, heavy)])
    for l in range(L):
        k[l].normal_(generator=gen)
        v[l].normal_(generator=gen)
        flat = k[l].view(P * PAGE, H, D)
        spans, heavy = places[l % 2]
        if spans is not None:
            flat[spans] = (flat[spans].float() + 1.5 * lean[l]).to(torch.bfloat16)
        flat[heavy] *= 3.0
    q = None
    if W:
        q = torch.randn((L, B, Hq, W, D), generator=gen, device=DEVICE)
        q += 2.0 * lean.repeat_interleave(Hq // H, dim=1)[:, None, :, None, :]
        q = q.to(torch.bfloat16)
    fresh = torch.from_numpy(fresh).to(DEVICE)
    live = fresh.clone()
    st = dict(static=False, case=case, k=k, v=v, q=q, fresh=fresh, live=live, table=live[:B * stride].view(B, stride),
              lens=live[B * stride:], dst=torch.from_numpy(dst).to(DEVICE), n_src=n_src, ext=None,
              comp=binding.AmsCompressor(cfg, DEVICE))
    if case["carried"]:  # the kept tokens of the event before come first; the appended ones start without credit
        st["comp"].ema_state[..., :case["budget"]] = _scores((L, B, H, case["budget"]), gen)
    if case["scorer"] == "external":
        st["ext"] = _scores((L, B, H, case["cap"]), gen)
    if case["scorer"] == "expected":
        mean = 2.0 * lean.repeat_interleave(Hq // H, dim=1)[:, None] + 0.1 * torch.randn((L, B, Hq, D), generator=gen, device=DEVICE)
        cov = torch.empty((L, B, Hq, D, D), dtype=torch.bfloat16, device=DEVICE)
        for l in range(L):  # 0.5 I and eight directions, the one of the queries among them
            u = torch.nn.functional.normalize(torch.randn((B, Hq, 8, D), generator=gen, device=DEVICE), dim=-1)
            u[:, :, 0] = lean[l].repeat_interleave(Hq // H, dim=0)
            w = 0.5 + 3.5 * torch.rand((B, Hq, 8, 1), generator=gen, device=DEVICE)
            cov[l] = (0.5 * torch.eye(D, device=DEVICE) + (u * w).transpose(-1, -2) @ u).to(torch.bfloat16)
        st["comp"].set_query_stats(mean.contiguous(), cov)
    return st


def run(state):
    case = state["case"]
    if state["static"]:
        binding.select_static(state["cfg"], state["scores"], state["T"], case["budget"], case["segments"], state["keep"])
        return {"keep": state["keep"]}
    state["live"].copy_(state["fresh"])  # the loop's table and lengths of this event
    comp = state["comp"]
    comp.compress(state["k"], state["v"], state["table"], state["lens"], state["q"], case["budget"], case["segments"],
                  SCORERS[case["scorer"]], state["dst"], ext_scores=state["ext"])
    # All of the replacement pages, the new table and lengths, and the credit of every row.  Rows move as a whole: where two
    # tokens tie within rounding, the rows between them shift by one, which only "how many values differ" can tell, so bf16
    # rows come as 16-bit words; the credit comes at bf16 precision (the upper word of each value) for the same reason.
    return {"k": state["k"][:, state["n_src"]:].view(torch.int16), "v": state["v"][:, state["n_src"]:].view(torch.int16),
            "table": state["table"], "lens": state["lens"], "credit": comp.ema_state.view(torch.int16)[..., 1::2]}


def work(case):
    """K read once (V too where the score uses value norms), caller's scores, query statistics, credit read and written,
    kept K and V rows read and written; two operations per multiply-add of the scores' products."""
    if case["scorer"] == "static":
        return {"bytes": case["kv_heads"] * (case["t_max"] + case["budget"]) * 4, "flops": 0}
    units, tokens = case["layers"] * case["kv_heads"], sum(_lens(case))
    n = units * tokens
    bytes_ = case["batch"] * units * case["budget"] * 1024
    flops = 0
    group = case["q_heads"] // case["kv_heads"]
    if case["beta"] != 1.0:
        bytes_ += 8 * n
    if case["scorer"] == "external":
        bytes_ += 4 * n
    else:
        bytes_ += 256 * n
    if case["window"]:
        flops += 2 * D * group * case["window"] * n
        bytes_ += case["layers"] * case["batch"] * case["q_heads"] * case["window"] * D * 2
    if case["scorer"] == "expected":
        flops += 2 * (D * D + 2 * D) * group * n
        bytes_ += 256 * n + case["layers"] * case["batch"] * case["q_heads"] * (D * 4 + D * D * 2)
    if case["scorer"] == "keydiff":
        flops += 6 * D * n
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Given scores, every result is an integer or a moved byte.  Scores in another order of summation (measured: relative
    noise of 1e-7 to 1e-6 on them) tip near-ties: up to 1.4e-3 of the output words then differ."""
    if case["scorer"] in ("static", "external"):
        return "exact"
    return {"rel": 0.0, "differ": 0.005}
