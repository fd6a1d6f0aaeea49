"""Window scores of up to 63 query rows where logits are large but finite: beyond 2^31 the rounding of a product in fp32 is more than an
exponent of fp32 can hold, and a row's logits may all lie below any fixed reference.  The likeliest token of a row then has all of
its probability, in fp32 as in the oracle's fp64, so scores stay within the 1e-3 of ordinary logits."""
import pytest
import torch

import oracle
from helpers import HostSnapshot, assert_scores_close, gpu_event
from paper_2605_23200_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
T = 700


@pytest.mark.parametrize("kind", ["large", "all_below"])
@pytest.mark.parametrize("heads,window", [((28, 4), 1), ((28, 4), 2), ((32, 8), 8), ((32, 8), 10)])
def test_window_scores_of_large_logits(heads, window, kind):
    wl = inputs.CONFIGS[2].scaled(n_layers=1, batch=1, n_q_heads=heads[0], n_kv_heads=heads[1], window=window, seq_len_min=T,
                                  seq_len_max=T, budget=64, resident_layers=0)
    cache = inputs.make_cache(wl, DEV)
    if kind == "large":
        cache.obs_queries *= 2.0 ** 40  # logits of 1e12 to 1e14, far apart
    else:
        cache.k_pages[..., 0].uniform_(1.25, 2.0, generator=torch.Generator(DEV).manual_seed(7))
        page = int(cache.block_table[0, 11])
        cache.k_pages[0, page, 5, :, 0] = 1.0  # the likeliest token
        cache.obs_queries.zero_()
        cache.obs_queries[..., 0] = -(2.0 ** 110)  # logits of -1e32 to -3e32
    comp = binding.AmsCompressor(binding.config_for(wl), DEV)
    snap = HostSnapshot(cache)
    got = gpu_event(comp, cache, inputs.alloc_dst_pages(cache)).scores.cpu().numpy()
    G = wl.group
    for h in range(wl.n_kv_heads):
        want = oracle.score_tova(snap.k, 0, h, snap.table[0], T, snap.q[0, 0, h * G:(h + 1) * G], G, window, True)
        assert_scores_close(got[0, 0, h, :T], want, rtol=1e-3)
