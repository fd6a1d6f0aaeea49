"""Tensor-core window scorer by its number of 128-row query blocks: products go to four accumulator slots in turn, a tile's blocks meet
across warpgroups; several units per block, ragged lengths whose last tile holds few tokens."""
import pytest

from paper_2605_23200_b200 import inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,heads", [(16, (32, 8)), (33, (16, 4)), (31, (64, 8)), (33, (64, 8)), (48, (32, 4)), (50, (16, 2)), (64, (8, 1))])
@pytest.mark.parametrize("lens", [(257, 1300), (2050, 2050)])
def test_scores_by_query_blocks(window, heads, lens):
    """64, 132, 248, 264, 384, 400 and 512 query rows: one to four blocks, full and padded."""
    wl = inputs.CONFIGS[0].scaled(n_layers=2, batch=3, n_q_heads=heads[0], n_kv_heads=heads[1], seq_len_min=lens[0], seq_len_max=lens[1], budget=200,
                                  window=window, resident_layers=0)
    _check_scorer(wl, rtol=1e-3, sample_units=[(0, 0, 0), (1, 1, heads[1] - 1), (1, 2, 0)])
