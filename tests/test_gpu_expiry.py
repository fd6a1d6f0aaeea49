"""A wait inside a scorer, or of the row moves, that runs out: every role of every block returns with its copies landed, the event
reports AMS_ERR_TIMEOUT and leaves pages, table and lengths alone (a scorer also the credit), and the next event on the handle is exact.
The wait is made to run out by construction (for an arrival that nobody makes)."""
import pytest
import torch

import oracle
from helpers import HostSnapshot, compare_event, gpu_event, params_of
from paper_2605_23200_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    dict(cfg=3, n_layers=1, batch=1, seq_len_min=4096, seq_len_max=4096),                                          # key-only, a cluster per unit
    dict(cfg=3, n_layers=3, batch=4, seq_len_min=9000, seq_len_max=9001),                                          # key-only, groups over the whole device
    dict(cfg=2, n_q_heads=32, n_kv_heads=8, window=1, n_layers=1, batch=1, seq_len_min=4096, seq_len_max=4096),    # 4 rows, a cluster per unit
    dict(cfg=2, n_q_heads=28, n_kv_heads=4, window=1, n_layers=2, batch=5, seq_len_min=3000, seq_len_max=9001),    # 7 rows, whole device
    dict(cfg=2, n_q_heads=28, n_kv_heads=4, window=2, n_layers=2, batch=5, seq_len_min=3000, seq_len_max=9001),    # 14 rows
    dict(cfg=2, n_q_heads=32, n_kv_heads=8, window=8, n_layers=2, batch=3, seq_len_min=3000, seq_len_max=9001),    # 32 rows
    dict(cfg=2, n_q_heads=32, n_kv_heads=8, window=32, n_layers=2, batch=2, seq_len_min=3000, seq_len_max=5000),   # 128 rows
    dict(cfg=1, n_q_heads=32, n_kv_heads=8, window=0, n_layers=2, batch=2, seq_len_min=3000, seq_len_max=5000, scorer_id=inputs.SCORER_EXPECTED),
]


@pytest.mark.parametrize("polls", [1, 300])
@pytest.mark.parametrize("kw", CASES)
def test_a_wait_that_runs_out_inside_a_scorer(kw, polls):
    kw = dict(kw)
    wl = inputs.CONFIGS[kw.pop("cfg")].scaled(budget=512, resident_layers=0, **kw)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    if wl.scorer_id == inputs.SCORER_EXPECTED:
        mean, cov = inputs.make_query_stats(cache)
        comp.set_query_stats(mean, cov, 1e-2)
    comp.ema_state.uniform_(0.0, 1e-3)
    dst = inputs.alloc_dst_pages(cache)
    own = [cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, comp.ema_state]
    before = [t.clone() for t in own]
    views = comp.make_debug_views(wl.batch, wl.budget)
    views.prev_kept = torch.full((wl.batch,), 64, dtype=torch.int32, device=DEV)
    views.retained_iou = iou = torch.zeros((wl.n_layers, wl.batch, wl.n_kv_heads), device=DEV)
    comp.expire_event(polls)
    comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, cache.obs_queries if wl.window else None, wl.budget,
                  wl.n_segments, wl.scorer_id, torch.from_numpy(dst).to(DEV), dbg=views)
    assert comp.status(check=False)[0] == binding.AMS_ERR_TIMEOUT
    for t, b in zip(own, before):
        raw = torch.int16 if t.element_size() == 2 else torch.int32
        assert torch.equal(t.view(raw), b.view(raw))
    assert not bool(views.keep_idx.any()) and not bool(views.n_segments.any()) and not bool(iou.any())
    snap = HostSnapshot(cache)
    credit0 = comp.ema_state.cpu().numpy()
    dbg = gpu_event(comp, cache, dst)
    units = [(l, b, h) for l in {0, wl.n_layers - 1} for b in {0, wl.batch - 1} for h in {0, wl.n_kv_heads - 1}]
    compare_event(snap, cache, comp, dbg, dst, credit0, dbg.scores.cpu().numpy(), units=units)
    with pytest.raises(binding.AmsError):
        comp.expire_event(0)


JOINT = dict(n_layers=37, batch=12, seq_len_min=520, seq_len_max=900, budget=460)  # 1776 units: selection and moves in one launch


@pytest.mark.parametrize("kw,launches", [
    (dict(cfg=3, n_q_heads=32, n_kv_heads=4, l_max=256, **JOINT), 3),                                            # key-only scores
    (dict(cfg=2, n_q_heads=28, n_kv_heads=4, window=1, **JOINT), 3),                                             # 7 rows
    (dict(cfg=2, n_q_heads=32, n_kv_heads=4, window=16, **JOINT), 4),                                            # 128 rows
    (dict(cfg=2, n_q_heads=28, n_kv_heads=4, window=1, n_layers=2, batch=5, seq_len_min=700, seq_len_max=3000, budget=512), 4),  # moves of their own
])
def test_a_scorer_that_gave_up_without_views(kw, launches):
    """Nothing changes, and the next event on the handle, without views too, is the oracle's."""
    kw = dict(kw)
    wl = inputs.CONFIGS[kw.pop("cfg")].scaled(resident_layers=0, **kw)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    comp.ema_state.uniform_(0.0, 1e-3)
    dst_np = inputs.alloc_dst_pages(cache)
    dst = torch.from_numpy(dst_np).to(DEV)
    own = [cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, comp.ema_state]
    before = [t.clone() for t in own]
    comp.expire_event(3)
    comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, cache.obs_queries if wl.window else None, wl.budget,
                  wl.n_segments, wl.scorer_id, dst)
    assert comp.last_launch_count == launches
    assert comp.status(check=False)[0] == binding.AMS_ERR_TIMEOUT
    for t, b in zip(own, before):
        raw = torch.int16 if t.element_size() == 2 else torch.int32
        assert torch.equal(t.view(raw), b.view(raw))
    ext = torch.rand((wl.n_layers, wl.batch, wl.n_kv_heads, wl.max_seq_len), device=DEV)
    snap, credit = HostSnapshot(cache), comp.ema_state.cpu().numpy()
    comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments,
                  binding.AMS_SCORER_EXTERNAL, dst, ext_scores=ext)
    comp.status()
    oracle.compress(snap.k, snap.v, snap.table, snap.lens, None, credit, wl.budget, params_of(wl), oracle.SCORER_EXTERNAL, dst_np,
                    ext_scores=ext.cpu().numpy(), threads=8)
    assert (inputs.as_u16(cache.k_pages) == snap.k).all() and (inputs.as_u16(cache.v_pages) == snap.v).all()
    assert (cache.block_table.cpu().numpy() == snap.table).all() and (cache.seq_lens.cpu().numpy() == snap.lens).all()
    assert wl.ema_beta == 1.0 or (comp.ema_state.cpu().numpy() == credit).all()


@pytest.mark.parametrize("polls", [1, 300])
def test_a_wait_of_the_moves_that_runs_out(polls):
    """External scores, so that only the moves of the joint launch wait: table, lengths and live pages stay, and the next event is exact."""
    wl = inputs.CONFIGS[2].scaled(resident_layers=0, n_q_heads=28, n_kv_heads=4, **JOINT)
    cache = inputs.make_cache(wl, DEV)
    short = 3
    cache.seq_lens[short] = wl.budget - 5  # within the budget: its moves have nothing to wait for
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    dst_np = inputs.alloc_dst_pages(cache)
    dst = torch.from_numpy(dst_np).to(DEV)
    ext = torch.rand((wl.n_layers, wl.batch, wl.n_kv_heads, wl.max_seq_len), device=DEV)
    args = (cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments, binding.AMS_SCORER_EXTERNAL, dst)
    before = [t.clone() for t in (cache.block_table, cache.seq_lens, cache.k_pages, cache.v_pages)]
    comp.expire_event(polls)
    comp.compress(*args, ext_scores=ext)
    assert comp.last_launch_count == 2
    rc, detail = comp.status(check=False)
    assert rc == binding.AMS_ERR_TIMEOUT and detail[1] % wl.n_kv_heads == 0 and detail[3] == wl.n_kv_heads + 1
    assert torch.equal(cache.block_table, before[0]) and torch.equal(cache.seq_lens, before[1])
    assert torch.equal(cache.k_pages.view(torch.int16), before[2].view(torch.int16))  # (no part moved a row)
    assert torch.equal(cache.v_pages.view(torch.int16), before[3].view(torch.int16))
    snap, credit = HostSnapshot(cache), comp.ema_state.cpu().numpy()
    comp.compress(*args, ext_scores=ext)
    comp.status()
    oracle.compress(snap.k, snap.v, snap.table, snap.lens, None, credit, wl.budget, params_of(wl), oracle.SCORER_EXTERNAL, dst_np,
                    ext_scores=ext.cpu().numpy(), threads=8)
    assert (inputs.as_u16(cache.k_pages) == snap.k).all() and (inputs.as_u16(cache.v_pages) == snap.v).all()
    assert (cache.block_table.cpu().numpy() == snap.table).all() and (cache.seq_lens.cpu().numpy() == snap.lens).all()
    assert (comp.ema_state.cpu().numpy() == credit).all()
