"""Selection kernel at the edges of its search forms, bit-exact against the oracle: segments of exactly one register piece
(256 tokens) and one more, several batches of long segments, score ranges beyond the first histogram, ties across the
threshold, zero and negative scores, and sequences whose pieces outnumber the table of best rejected keys."""
import numpy as np
import pytest
import torch

from helpers import HostSnapshot, compare_event, gpu_event
from paper_2605_23200_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _scores(kind, shape, rng):
    if kind == "wide":      # sixty octaves: most thresholds lie far below the largest score of their segment
        x = np.exp(rng.uniform(-40.0, 2.0, size=shape))
    elif kind == "tiny":    # subnormal and zero scores
        x = rng.random(shape) * 1e-40
        x[rng.random(shape) < 0.3] = 0.0
    elif kind == "signed":  # like a cosine: both signs, near zero in between
        x = rng.standard_normal(shape) * 0.1
    elif kind == "steps":   # few distinct values: ties across nearly every threshold
        x = rng.integers(1, 6, size=shape) * 0.125
    elif kind == "negative_nan":
        x = -np.exp(rng.standard_normal(shape))
        x[rng.random(shape) < 0.05] = np.nan
    else:
        x = np.exp(1.5 * rng.standard_normal(shape))
    return x.astype(np.float32)


CASES = [
    ("plain", dict(seq_len_min=2560, seq_len_max=2560, l_max=256, n_segments=1, budget=640)),      # ten pieces of exactly 256
    ("plain", dict(seq_len_min=2570, seq_len_max=2570, l_max=257, n_segments=1, budget=640)),      # ten of 257: the long form
    ("wide", dict(seq_len_min=4097, seq_len_max=4097, budget=700)),
    ("wide", dict(seq_len_min=9000, seq_len_max=9000, budget=1500, l_max=2000, n_segments=5)),
    ("tiny", dict(seq_len_min=3000, seq_len_max=3000, budget=900)),
    ("tiny", dict(seq_len_min=6000, seq_len_max=6000, budget=900, l_max=3000, n_segments=4)),
    ("signed", dict(seq_len_min=5001, seq_len_max=5001, budget=512)),
    ("signed", dict(seq_len_min=20000, seq_len_max=20000, budget=2000, l_max=4096, n_segments=16, ema_beta=1.0)),
    ("steps", dict(seq_len_min=5000, seq_len_max=5000, budget=1111)),
    ("steps", dict(seq_len_min=30000, seq_len_max=30000, budget=3000, l_max=300, n_segments=3, batch=1)),  # two batches of long segments
    ("negative_nan", dict(seq_len_min=3000, seq_len_max=3000, budget=2990, n_last=40)),
    ("negative_nan", dict(seq_len_min=8000, seq_len_max=8000, budget=7900, l_max=1000, n_last=40)),
    ("plain", dict(seq_len_min=60000, seq_len_max=60000, budget=6000, l_max=64, n_segments=10, batch=1, n_kv_heads=2, n_q_heads=8)),
    ("plain", dict(seq_len_min=131072, seq_len_max=131072, budget=300, l_max=0, n_segments=1, batch=1, n_kv_heads=1, n_q_heads=4)),
    ("plain", dict(seq_len_min=700, seq_len_max=1500, budget=400, batch=24, n_layers=5)),           # many units: the narrow blocks
]


@pytest.mark.parametrize("kind,kw", CASES)
def test_search_forms_match_the_oracle(kind, kw):
    base = dict(n_layers=1, batch=2, resident_layers=0)
    base.update(kw)
    wl = inputs.CONFIGS[0].scaled(**base)
    cache = inputs.make_cache(wl, DEV)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    ext = _scores(kind, (wl.n_layers, wl.batch, wl.n_kv_heads, wl.max_seq_len), np.random.default_rng(99))
    snap = HostSnapshot(cache)
    credit0 = comp.ema_state.cpu().numpy()
    dst = inputs.alloc_dst_pages(cache)
    dbg = gpu_event(comp, cache, dst, inputs.SCORER_EXTERNAL, torch.from_numpy(ext).to(DEV))
    compare_event(snap, cache, comp, dbg, dst, credit0, ext)
