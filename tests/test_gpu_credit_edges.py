"""Credit rows that say nothing: a restored credit that is negative or not a number throughout, or infinite anywhere, is left out of the mass, and with
ema_beta = 0 the unit then has no mass at all (every threshold of the cut search is 0, every share of the budget too)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import HostSnapshot, compare_event, gpu_event
from paper_2605_23200_b200 import binding, inputs

SHAPES = [
    dict(seq_len_min=1500, seq_len_max=1500, budget=384),
    dict(seq_len_min=700, seq_len_max=1777, budget=600, n_segments=32, l_min=1, q_min=2, batch=4),        # a first segment of one token
    dict(seq_len_min=9001, seq_len_max=9001, budget=1024, batch=1, l_max=4096),                           # a long segment
    dict(seq_len_min=40000, seq_len_max=40000, budget=2000, batch=1, n_layers=1, n_segments=16, l_max=0), # more than 1024 windows, no split
]


def _event(kw, beta, fill):
    base = dict(n_layers=2, batch=2)
    base.update(kw)
    wl = inputs.CONFIGS[0].scaled(resident_layers=0, ema_beta=beta, **base)
    cache = inputs.make_cache(wl, "cuda:0")
    comp = binding.AmsCompressor(binding.config_for(wl), "cuda:0")
    rng = np.random.default_rng(17)
    ext = np.exp(2.0 * rng.standard_normal((wl.n_layers, wl.batch, wl.n_kv_heads, wl.max_seq_len))).astype(np.float32)
    if fill == "one":
        comp.ema_state.uniform_(0.0, 1e-3)
        comp.ema_state[..., 300] = float("inf")
    else:
        comp.ema_state.fill_(fill)
    snap, credit0 = HostSnapshot(cache), comp.ema_state.cpu().numpy()
    dst = inputs.alloc_dst_pages(cache)
    dbg = gpu_event(comp, cache, dst, inputs.SCORER_EXTERNAL, torch.from_numpy(ext).to("cuda:0"))
    return wl, cache, comp, snap, credit0, dst, dbg, ext


@pytest.mark.gpu
@pytest.mark.parametrize("beta", [0.0, 0.9])
@pytest.mark.parametrize("kw", SHAPES)
def test_negative_credit(kw, beta):
    wl, cache, comp, snap, credit0, dst, dbg, ext = _event(kw, beta, -1.0)
    res = compare_event(snap, cache, comp, dbg, dst, credit0, ext)
    if beta == 0.0 and wl.l_min == 16 and wl.l_max == 256:
        assert all(np.ptp(r.quotas) <= 1 for r in res.values())  # equal shares


@pytest.mark.gpu
@pytest.mark.parametrize("fill", [float("nan"), float("inf"), "one"])
@pytest.mark.parametrize("beta", [0.0, 0.9])
@pytest.mark.parametrize("kw", SHAPES)
def test_credit_that_is_not_finite(kw, beta, fill):
    """Kept rows as with a negative credit; the credit itself stays what it is.  "one": one infinite token in each unit."""
    wl, cache, comp, snap, credit0, dst, dbg, ext = _event(kw, beta, fill)
    prm = oracle.Params(wl.n_segments, wl.l_min, wl.l_max, wl.q_min, wl.n_sink, wl.n_last, wl.ema_lambda, beta, wl.eps)
    res = oracle.compress(snap.k, snap.v, snap.table, snap.lens, None, np.full_like(credit0, -1.0), wl.budget, prm,
                          oracle.SCORER_EXTERNAL, dst, ext_scores=ext, threads=8)
    keep = dbg.keep_idx.cpu().numpy()
    for u, r in res.items():
        assert (keep[u] == r.keep_idx).all(), u
    assert (inputs.as_u16(cache.k_pages) == snap.k).all() and (inputs.as_u16(cache.v_pages) == snap.v).all()
    if fill != "one":
        assert not bool(torch.isfinite(comp.ema_state[..., :wl.budget]).any())


def test_oracle_shares_equally_where_there_is_no_mass():
    q = oracle.quotas(np.zeros(100, np.uint64), [0, 20, 30, 70, 100], 2, 50)
    assert q.tolist() == [14, 10, 13, 13]
