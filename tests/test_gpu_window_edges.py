"""Window scorers below 64 query rows at the edges of their streams of tiles, against the oracle (scores and mass within 1e-3,
selection exact): every padded row count, fewer tiles than warps, one token past a tile, a page or a slice, windows longer than
a tile, and more (unit, slice) pairs than blocks, so that a block's stream runs on from one unit into another."""
import pytest

from paper_2605_23200_b200 import inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu

CASES = [
    dict(n_q_heads=8, n_kv_heads=8, window=1, seq_len_min=33, seq_len_max=33, budget=20),           # 1 row, three tiles
    dict(n_q_heads=28, n_kv_heads=4, window=1, seq_len_min=513, seq_len_max=1025, batch=5),         # 7 rows, one token past slices
    dict(n_q_heads=16, n_kv_heads=8, window=8, seq_len_min=700, seq_len_max=700),                   # 16 rows
    dict(n_q_heads=16, n_kv_heads=8, window=9, seq_len_min=40, seq_len_max=64, budget=24, batch=3), # 18 rows in 32, masked tiles only
    dict(n_q_heads=32, n_kv_heads=8, window=8, seq_len_min=600, seq_len_max=1601, batch=24, n_layers=4), # 32 rows, more work than blocks
    dict(n_q_heads=32, n_kv_heads=8, window=9, seq_len_min=1200, seq_len_max=1200),                 # 36 rows in 64
    dict(n_q_heads=28, n_kv_heads=4, window=9, seq_len_min=2049, seq_len_max=2049),   # 63 rows
    dict(n_q_heads=28, n_kv_heads=4, window=1, seq_len_min=400, seq_len_max=3000, batch=40, n_layers=6),
]


@pytest.mark.parametrize("kw", CASES)
def test_window_scores_match_the_oracle(kw):
    base = dict(n_layers=1, batch=2, budget=256, resident_layers=0)
    base.update(kw)
    wl = inputs.CONFIGS[2].scaled(**base)
    units = [(l, b, h) for l in {0, wl.n_layers - 1} for b in {0, wl.batch // 2, wl.batch - 1} for h in {0, wl.n_kv_heads - 1}]
    _check_scorer(wl, sample_units=units)
