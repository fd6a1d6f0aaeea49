"""Sequences within the budget cost the scorers that share units between groups of blocks nothing: the same events with and
without them take the same time, and the scores of what is compressed match the oracle."""
import pytest
import torch

from paper_2605_23200_b200 import binding, inputs
from test_gpu_parity import _check_scorer

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _scorer_ms(cfg, batch, skip, **kw):
    wl = inputs.CONFIGS[cfg].scaled(n_layers=8, batch=batch, seq_len_min=6400, seq_len_max=6400, budget=512, resident_layers=0, **kw)
    cache = inputs.make_cache(wl, DEV)
    cache.seq_lens[[b for b in range(batch) if skip(b)]] = wl.budget
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    comp.set_profiling(True)
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)
    table0, lens0 = cache.block_table.clone(), cache.seq_lens.clone()
    times = []
    for _ in range(9):
        cache.block_table.copy_(table0)
        cache.seq_lens.copy_(lens0)
        comp.compress(cache.k_pages, cache.v_pages, cache.block_table, cache.seq_lens, cache.obs_queries if wl.window else None, wl.budget,
                      wl.n_segments, wl.scorer_id, dst)
        times.append(comp.kernel_times_ms()["score_phase1"])
    comp.status()
    return sorted(times)[len(times) // 2]


@pytest.mark.parametrize("skip", ["every_other", "first_eight"])
@pytest.mark.parametrize("kw", [dict(cfg=3, n_q_heads=32, n_kv_heads=8), dict(cfg=2, n_q_heads=32, n_kv_heads=8, window=1),
                                dict(cfg=2, n_q_heads=32, n_kv_heads=8, window=8)])
def test_skipped_sequences_take_no_time(kw, skip):
    """Half of the device idle would be a factor of two; other differences (lengths read, pages elsewhere) are a few per cent."""
    alone = _scorer_ms(batch=8, skip=lambda b: False, **kw)
    among = _scorer_ms(batch=16, skip=lambda b: b % 2 == 1 if skip == "every_other" else b < 8, **kw)
    assert among < 1.3 * alone, (among, alone)


@pytest.mark.parametrize("batch,budget", [(1, 400), (7, 900), (40, 1024), (70, 1400)])
@pytest.mark.parametrize("cfg", [2, 3])
def test_scores_among_skipped_sequences(cfg, batch, budget):
    """Ragged lengths from 300 to 1500, so that up to nine sequences in ten are skipped: more sequences than lanes, runs of them."""
    wl = inputs.CONFIGS[cfg].scaled(n_layers=2, batch=batch, n_q_heads=14, n_kv_heads=2, seq_len_min=300, seq_len_max=1500, budget=budget,
                                    resident_layers=0)
    _check_scorer(wl, rtol=1e-3, atol=1e-5 if cfg == 3 else 0.0)
