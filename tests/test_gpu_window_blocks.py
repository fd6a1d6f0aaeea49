"""Tensor-core window scorer by its number of 128-row query blocks: products go to four accumulator slots in turn, a tile's blocks meet
across warpgroups; several units per block, ragged lengths whose last tile holds few tokens."""
import numpy as np
import pytest
import torch

from helpers import gpu_event
from paper_2605_23200_b200 import binding, inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,heads", [(16, (32, 8)), (33, (16, 4)), (31, (64, 8)), (33, (64, 8)), (48, (32, 4)), (50, (16, 2)), (64, (8, 1))])
@pytest.mark.parametrize("lens", [(257, 1300), (2050, 2050)])
def test_scores_by_query_blocks(window, heads, lens):
    """64, 132, 248, 264, 384, 400 and 512 query rows: one to four blocks, full and padded.  The tolerance is four times the 5e-6 that
    fp32 gives where logits stay below 64 (log2): half a unit each of the exponential's argument and of a row's reference 1.3e-6,
    ex2.approx twice 5e-7, sums 5e-7, products 1e-6."""
    wl = inputs.CONFIGS[0].scaled(n_layers=2, batch=3, n_q_heads=heads[0], n_kv_heads=heads[1], seq_len_min=lens[0], seq_len_max=lens[1], budget=200,
                                  window=window, resident_layers=0)
    _check_scorer(wl, rtol=2e-5, sample_units=[(0, 0, 0), (1, 1, heads[1] - 1), (1, 2, 0)])


@pytest.mark.parametrize("tail", [False, True])
@pytest.mark.parametrize("window", [24, 40])
def test_row_sums_of_many_chunks(window, tail):
    """192 and 320 rows (two and three query blocks), 131072 tokens, a block to a unit: a thread adds up to 2048 chunks of 32 columns.
    Every chunk has the same sum (the keys repeat every 32 tokens), so that without compensation, with its sign turned or, where the
    last tokens raise the maximum by ten octaves, without its rescaling the rounding of a row's sum adds up to 6e-6 and more (emulated;
    with it 2e-7).  What else may differ: the fused multiply-add before the exponential and the reference of a row (|.| < 32 and
    < 16 in log2, half a unit each: 6.6e-7 and 3.3e-7), the rounded scale (5e-7), ex2.approx twice (2.4e-7 each) and sums of 32
    and of the rows (2e-7 each): 3e-6 in all."""
    T, H = 131072, 4
    wl = inputs.CONFIGS[0].scaled(n_layers=37, batch=1, n_q_heads=8 * H, n_kv_heads=H, seq_len_min=T, seq_len_max=T, budget=512, window=window,
                                  resident_layers=0)
    cache = inputs.make_cache(wl, "cuda:0")
    comp = binding.AmsCompressor(binding.config_for(wl, causal_window=0), "cuda:0")
    chunks = np.stack([np.random.default_rng(s).choice(np.arange(-1.5, 0.25, 0.25), 32) for s in (1, 29, 33, 36)], 1)  # [32][H]
    chunks[0] = 0.0
    keys = torch.from_numpy(np.tile(chunks, (T // 32, 1))).cuda()
    if tail:
        keys[-512:] += 5.0
    cache.k_pages.zero_()
    cache.k_pages[:, cache.block_table[0, :T // 16].long(), :, :, 0] = keys.view(T // 16, 16, H).to(torch.bfloat16)
    cache.obs_queries.zero_()
    cache.obs_queries[..., 0] = 16.0
    got = gpu_event(comp, cache, inputs.alloc_dst_pages(cache)).scores.double()
    want = torch.softmax(keys * (16.0 / 128 ** 0.5), 0).T  # fp64, the same for every row
    assert float(((got[:, 0] - want) / want).abs().max()) < 3e-6
