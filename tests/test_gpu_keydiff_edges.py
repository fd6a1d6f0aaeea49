"""Key-only scores, which groups of blocks compute together, at the edges of their split, against the oracle.  Both sides
accumulate in fp32 or better and the products are exact, so a score, a cosine in [-1, 1], differs by at most the rounding of
sums of 128 terms and of up to 70001 keys: within 1e-3 relative and 1e-5 absolute."""
import pytest
import torch

from paper_2605_23200_b200 import binding, inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    dict(n_q_heads=8, n_kv_heads=1, batch=1, seq_len_min=33, seq_len_max=33, budget=20),                 # one unit, three pages, the last with one token
    dict(n_q_heads=8, n_kv_heads=1, batch=1, seq_len_min=70001, seq_len_max=70001, budget=512),          # one unit over the whole chip
    dict(batch=3, seq_len_min=256, seq_len_max=257, budget=256),                                         # a sequence within the budget between others
    dict(batch=5, n_layers=2, seq_len_min=300, seq_len_max=9001, budget=290),                            # blocks without a page of the short ones
    dict(batch=40, n_layers=3, seq_len_min=900, seq_len_max=1100, budget=256),                           # more units than blocks
    dict(n_q_heads=28, n_kv_heads=4, batch=2, seq_len_min=30000, seq_len_max=32769, budget=512),         # fewer units than fit L2
    dict(n_q_heads=40, n_kv_heads=8, batch=3, n_layers=3, seq_len_min=16000, seq_len_max=16400, budget=512),  # several units per group
]


@pytest.mark.parametrize("kw", CASES)
def test_key_scores_match_the_oracle(kw):
    base = dict(n_layers=1, resident_layers=0)
    base.update(kw)
    wl = inputs.CONFIGS[3].scaled(**base)
    units = [(l, b, h) for l in {0, wl.n_layers - 1} for b in {0, wl.batch // 2, wl.batch - 1} for h in {0, wl.n_kv_heads - 1}]
    _check_scorer(wl, sample_units=units, rtol=1e-3, atol=1e-5)


def test_key_scores_repeat_exactly_and_replay_from_a_graph():
    wl = inputs.CONFIGS[3].scaled(n_layers=2, batch=6, seq_len_min=5000, seq_len_max=7000, budget=512, resident_layers=0)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)
    table0, lens0 = cache.block_table.clone(), cache.seq_lens.clone()
    dbg = comp.make_debug_views(wl.batch, wl.budget)

    def event():
        comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, None, wl.budget, wl.n_segments,
                      wl.scorer_id, dst, dbg=dbg)

    def result():
        comp.status()
        got = [dbg.scores.clone(), dbg.keep_idx.clone(), cache.block_table.clone()]
        cache.block_table.copy_(table0)
        cache.seq_lens.copy_(lens0)
        comp.ema_state.zero_()
        dbg.scores.zero_()
        dbg.keep_idx.zero_()
        return got

    event()
    want = result()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        event()
    for run in (event, graph.replay, graph.replay):
        run()
        for a, b in zip(result(), want):
            assert torch.equal(a, b)
