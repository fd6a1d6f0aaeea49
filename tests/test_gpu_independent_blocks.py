"""Scorers whose blocks do not wait for one another: scores against the oracle (1e-3, key scores 1e-5 absolute besides), the same bits
for a sequence alone and in a batch, no wait that could run out; and how far the default ones move with the batch."""
import pytest
import torch

import oracle
from helpers import HostSnapshot, assert_scores_close
from paper_2605_23200_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    dict(cfg=3, n_q_heads=8, n_kv_heads=4),
    dict(cfg=2, n_q_heads=8, n_kv_heads=2, window=1),    # 4 rows
    dict(cfg=2, n_q_heads=14, n_kv_heads=2, window=2),   # 14 rows
    dict(cfg=2, n_q_heads=8, n_kv_heads=2, window=8),    # 32 rows
    dict(cfg=2, n_q_heads=8, n_kv_heads=2, window=15),   # 60 rows
]


def _scores(comp, cache, dst, first, count):
    """Scores of sequences [first, first + count) as a call of their own; the table is left as it was."""
    wl = cache.wl
    table, lens = cache.block_table[first:first + count].clone(), cache.seq_lens[first:first + count].clone()
    q = cache.obs_queries[:, first:first + count].contiguous() if wl.window else None
    views = comp.make_debug_views(count, wl.budget)
    comp.compress(cache.k_pages, cache.v_pages, table, lens, q, wl.budget, wl.n_segments, wl.scorer_id, dst[first:first + count].contiguous(), dbg=views)
    comp.status()
    return views.scores


@pytest.mark.parametrize("kw", CASES)
def test_independent_blocks(kw):
    kw = dict(kw)
    wl = inputs.CONFIGS[kw.pop("cfg")].scaled(n_layers=2, batch=5, seq_len_min=700, seq_len_max=6001, budget=256, resident_layers=0, **kw)
    cache = inputs.make_cache(wl, DEV)
    snap = HostSnapshot(cache)
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    dst = torch.from_numpy(inputs.alloc_dst_pages(cache)).to(DEV)
    shared = _scores(comp, cache, dst, 0, wl.batch), _scores(comp, cache, dst, 2, 1)
    comp.set_independent_blocks(True)
    comp.expire_event(1)  # no scorer of this kind waits: nothing runs out
    batch, alone = _scores(comp, cache, dst, 0, wl.batch), _scores(comp, cache, dst, 2, 1)
    T, G, key = int(snap.lens[2]), wl.group, wl.scorer_id == inputs.SCORER_KEYDIFF
    assert torch.equal(batch[:, 2, :, :T], alone[:, 0, :, :T])
    for b in (0, 2):
        n = int(snap.lens[b])
        for h in range(wl.n_kv_heads):
            if key:
                want = oracle.score_keydiff(snap.k, 1, h, snap.table[b], n)
            else:
                want = oracle.score_tova(snap.k, 1, h, snap.table[b], n, snap.q[1, b, h * G:(h + 1) * G], G, wl.window, True)
            assert_scores_close(batch[1, b, h, :n].cpu().numpy(), want, rtol=1e-3, atol=1e-5 if key else 0.0)
    # the default ones: sums of up to 6001 fp32 terms in another order, 2^-24 each, errors that add up like a random walk
    a, c = shared[0][:, 2, :, :T].double(), shared[1][:, 0, :, :T].double()
    assert float((a - c).abs().max()) <= 1e-5 * float(a.abs().max())
