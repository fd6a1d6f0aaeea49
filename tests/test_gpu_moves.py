"""Row moves: the kernel that selects and moves in one launch (many units of short segments, no views) and the one that only moves and
rewrites the table leave the same bytes, table, lengths and credit as an event with views, whose launches are separate and are
checked against the oracle elsewhere.  External scores, so that every value is determined."""
import numpy as np
import pytest
import torch

import oracle
from helpers import HostSnapshot, params_of
from paper_2605_23200_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _scores(wl, cap, seed=5):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn((wl.n_layers, wl.batch, wl.n_kv_heads, cap), generator=g, device=DEV).exp_()


def _compressor(wl, cap):
    cfg = binding.config_for(wl)
    cfg.max_seq_len = cap
    return binding.AmsCompressor(cfg, DEV)


def _event(wl, views, cap=0, seed=5):
    cap = cap or wl.max_seq_len
    cache = inputs.make_cache(wl, DEV)
    comp = _compressor(wl, cap)
    ext = _scores(wl, cap, seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    comp.ema_state.copy_(torch.rand(comp.ema_state.shape, generator=g, device=DEV))
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)
    dbg = comp.make_debug_views(wl.batch, wl.budget) if views else None
    for _ in range(1 if views else 2):  # (the second finds every sequence within the budget and changes nothing)
        comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments,
                      binding.AMS_SCORER_EXTERNAL, dst, ext_scores=ext, dbg=dbg)
        n = comp.last_launch_count
        comp.status()
    return cache, comp, n


@pytest.mark.parametrize("kw,launches", [
    # 12 units per SM (of 148) and more, budgets of 320 and more, from 16 units on of 400: one launch after the validation
    (dict(n_layers=80, batch=23, n_kv_heads=1, n_q_heads=1, seq_len_min=330, seq_len_max=700, budget=320), 2),  # one head
    (dict(n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=407), 2),   # part of a page left over
    (dict(n_layers=80, batch=23, n_kv_heads=1, n_q_heads=1, seq_len_min=401, seq_len_max=700, budget=400), 2),  # one head, one part
    (dict(n_layers=65, batch=11, n_kv_heads=3, n_q_heads=3, seq_len_min=200, seq_len_max=1000, budget=650), 2), # some within the budget
    (dict(n_layers=30, batch=2, n_kv_heads=40, n_q_heads=40, seq_len_min=500, seq_len_max=600, budget=431), 2), # more heads than a part's rows divide into
    (dict(n_layers=37, batch=12, n_kv_heads=4, n_q_heads=4, seq_len_min=514, seq_len_max=600, budget=513), 2),  # parts of 1024 rows and a few
    (dict(n_layers=37, batch=12, n_kv_heads=4, n_q_heads=4, seq_len_min=450, seq_len_max=600, budget=430, max_seq_len=65536), 2),  # 512 threads
    (dict(n_layers=37, batch=6, n_kv_heads=8, n_q_heads=8, seq_len_min=1500, seq_len_max=1700, budget=1536), 2),
    # few units, little to move, much to move in many heads, or segments above a piece: moves of their own, with the table
    (dict(n_layers=37, batch=6, n_kv_heads=8, n_q_heads=8, seq_len_min=1500, seq_len_max=1700, budget=1537), 3),
    (dict(n_layers=5, batch=5, n_kv_heads=71, n_q_heads=71, seq_len_min=300, seq_len_max=900, budget=407), 3),
    (dict(n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=327), 3),
    (dict(n_layers=80, batch=23, n_kv_heads=1, n_q_heads=1, seq_len_min=330, seq_len_max=700, budget=319), 3),
    (dict(n_layers=30, batch=2, n_kv_heads=40, n_q_heads=40, seq_len_min=500, seq_len_max=600, budget=337), 3),
    (dict(n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=319), 3),
    (dict(n_layers=2, batch=3, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=257), 3),
    (dict(n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=407, l_max=600), 3),
    (dict(n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=300, seq_len_max=900, budget=327, l_max=600), 3),
])
def test_event_without_views_equals_event_with_views(kw, launches):
    kw = dict(kw)
    cap = kw.pop("max_seq_len", 0)
    wl = inputs.CONFIGS[2].scaled(resident_layers=0, **kw)
    a, ca, _ = _event(wl, True, cap)
    b, cb, n = _event(wl, False, cap)
    assert n == launches
    assert torch.equal(a.k_pages.view(torch.int16), b.k_pages.view(torch.int16))
    assert torch.equal(a.v_pages.view(torch.int16), b.v_pages.view(torch.int16))
    assert torch.equal(a.block_table, b.block_table) and torch.equal(a.seq_lens, b.seq_lens)
    assert torch.equal(ca.ema_state, cb.ema_state)
    assert int((b.seq_lens == wl.budget).sum()) > 0


@pytest.mark.parametrize("shortest,budget,launches", [(420, 407, 2), (400, 327, 3)])
def test_bad_page_is_skipped_in_the_joint_launch(shortest, budget, launches):
    """A sequence with a page outside the pool keeps its row and length; the others are compressed (with the smaller budget in separate
    launches)."""
    wl = inputs.CONFIGS[2].scaled(resident_layers=0, n_layers=37, batch=9, n_kv_heads=8, n_q_heads=8, seq_len_min=shortest, seq_len_max=900,
                                  budget=budget)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    ext = torch.rand((wl.n_layers, wl.batch, wl.n_kv_heads, wl.max_seq_len), device=DEV)
    cache.block_table[4, 3] = cache.k_pages.shape[1]
    table, lens = cache.block_table.clone(), cache.seq_lens.clone()
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)
    comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments,
                  binding.AMS_SCORER_EXTERNAL, dst, ext_scores=ext)
    assert comp.last_launch_count == launches
    rc, detail = comp.status(check=False)
    assert rc == binding.AMS_ERR_INVALID_ARG and detail[1:4] == [4, 3, cache.k_pages.shape[1]]
    assert torch.equal(cache.block_table[4], table[4]) and cache.seq_lens[4] == lens[4]
    others = [b for b in range(wl.batch) if b != 4]
    assert (cache.seq_lens[others] == wl.budget).all() and torch.equal(cache.block_table[others][:, :dst.shape[1]], dst[others])


JOINT = dict(n_layers=37, batch=12, n_kv_heads=4, n_q_heads=4, seq_len_min=450, seq_len_max=900, budget=437)
APART = dict(n_layers=3, batch=5, n_kv_heads=4, n_q_heads=4, seq_len_min=450, seq_len_max=900, budget=437)


@pytest.mark.parametrize("kw,cap,launches", [(JOINT, 0, 2), (JOINT, 65536, 2), (APART, 0, 3)])
def test_event_without_views_equals_the_oracle_and_replays_from_a_graph(kw, cap, launches):
    """Rows, table, lengths and credit of a direct event against the oracle; the same event recorded into a CUDA graph gives the
    same bytes from restored inputs, twice (counters and page ids are written anew in each replay)."""
    wl = inputs.CONFIGS[2].scaled(resident_layers=0, **kw)
    cap = cap or wl.max_seq_len
    cache = inputs.make_cache(wl, DEV)
    comp = _compressor(wl, cap)
    ext = _scores(wl, cap)
    comp.ema_state.uniform_(0.0, 1e-3)
    dst_np = inputs.alloc_dst_pages(cache)
    dst = torch.from_numpy(dst_np).to(DEV)
    snap, credit = HostSnapshot(cache), comp.ema_state.cpu().numpy()
    inputs_before = [t.clone() for t in (cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, comp.ema_state)]

    def event():
        comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments,
                      binding.AMS_SCORER_EXTERNAL, dst, ext_scores=ext)

    def same_as_the_oracle():
        assert (inputs.as_u16(cache.k_pages) == snap.k).all() and (inputs.as_u16(cache.v_pages) == snap.v).all()
        assert (cache.block_table.cpu().numpy() == snap.table).all() and (cache.seq_lens.cpu().numpy() == snap.lens).all()
        assert (comp.ema_state.cpu().numpy() == credit).all()

    event()
    comp.status()
    assert comp.last_launch_count == launches
    oracle.compress(snap.k, snap.v, snap.table, snap.lens, None, credit, wl.budget, params_of(wl), oracle.SCORER_EXTERNAL, dst_np,
                    ext_scores=ext.cpu().numpy(), threads=8)
    same_as_the_oracle()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        event()
    for _ in range(2):
        for t, b in zip((cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, comp.ema_state), inputs_before):
            t.copy_(b)
        graph.replay()
        comp.status()
        same_as_the_oracle()
