"""Window scores up to 32 query rows, which groups of blocks compute together, at the edges of their split, against the oracle
(scores and mass within 1e-3: fp32 sums of bf16 products on both sides, selection exact on the library's own scores)."""
import pytest
import torch

from paper_2605_23200_b200 import binding, inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    dict(n_q_heads=8, n_kv_heads=1, window=1, batch=1, seq_len_min=33, seq_len_max=33, budget=20),          # 8 rows, three pages, the last with one token
    dict(n_q_heads=7, n_kv_heads=1, window=1, batch=1, seq_len_min=131072, seq_len_max=131072, budget=512), # 7 rows, the longest share of a block
    dict(n_q_heads=8, n_kv_heads=1, window=2, batch=1, seq_len_min=131065, seq_len_max=131065, budget=512), # 16 rows, the same
    dict(n_q_heads=16, n_kv_heads=4, window=3, batch=5, n_layers=2, seq_len_min=300, seq_len_max=9001, budget=290), # 12 rows, blocks without a page
    dict(n_q_heads=32, n_kv_heads=8, window=1, batch=3, seq_len_min=256, seq_len_max=257, budget=256),      # within the budget between others
    dict(n_q_heads=32, n_kv_heads=8, window=4, batch=40, n_layers=3, seq_len_min=900, seq_len_max=1100),    # 16 rows, more units than blocks
    dict(n_q_heads=32, n_kv_heads=8, window=7, batch=3, n_layers=3, seq_len_min=16000, seq_len_max=16400),  # 28 rows in 32, several units per group
    dict(n_q_heads=28, n_kv_heads=4, window=3, batch=2, seq_len_min=40000, seq_len_max=60001),              # 21 rows, fewer units than fit L2
]


@pytest.mark.parametrize("kw", CASES)
def test_window_scores_match_the_oracle(kw):
    base = dict(n_layers=1, budget=256, resident_layers=0)
    base.update(kw)
    wl = inputs.CONFIGS[2].scaled(**base)
    units = [(l, b, h) for l in {0, wl.n_layers - 1} for b in {0, wl.batch // 2, wl.batch - 1} for h in {0, wl.n_kv_heads - 1}]
    _check_scorer(wl, sample_units=units)


@pytest.mark.parametrize("heads,window", [((28, 4), 1), ((32, 8), 4), ((32, 8), 8)])
def test_window_scores_ignore_their_neighbours_queries(heads, window):
    """Rows are copied in eights, into the next unit's where there are fewer: nothing there may show."""
    wl = inputs.CONFIGS[2].scaled(n_layers=2, batch=2, n_q_heads=heads[0], n_kv_heads=heads[1], window=window, seq_len_min=700,
                                  seq_len_max=700, budget=64, resident_layers=0)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    table0, lens0 = cache.block_table.clone(), cache.seq_lens.clone()
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)

    def scores():
        cache.block_table.copy_(table0)
        cache.seq_lens.copy_(lens0)
        dbg = comp.make_debug_views(wl.batch, wl.budget)
        comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, cache.obs_queries, wl.budget, wl.n_segments,
                      wl.scorer_id, dst, dbg=dbg)
        comp.status()
        return dbg.scores[0, 0, 0, :700].clone()

    want = scores()
    G = heads[0] // heads[1]
    cache.obs_queries[0, 0, G:2 * G] = float("nan")
    assert torch.equal(scores(), want)
