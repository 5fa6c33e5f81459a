"""The allocation-free entry point at the edges of its pieces (two chunks long
at these sizes): one token, lengths around a chunk and around one and several
pieces, one-token chunks, and a chunk longer than the sequence, against the
fp64 oracle."""
import numpy as np
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache
from synth import gen
from synth.device import DeviceTrace

from .harness import OracleTrace, assert_scores_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,d,lag,lengths", [
    (2, 32, 16, (1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 95, 97, 300)),
    (3, 8, 1, (1, 2, 3, 9, 500)),
    (8, 128, 10, (19, 20, 21, 39, 41, 257, 270)),
    (4, 64, 300, (299, 300, 301, 599, 601, 950)),
    (1, 256, 1000, (700,)),
])
def test_piece_edges_against_the_oracle(H, d, lag, lengths):
    model = gen.TraceModel(0xE91C0300 + H * d + lag, num_layers=2, hidden=256, num_kv_heads=H, head_dim=d, band_a=(0,),
                           band_b=(1,))
    n_max = max(lengths)
    cache = KVCache(E.EPIKV_LAYOUT_PAGED, 2, H, d, max_seqs=1, max_tokens=n_max)
    dt = DeviceTrace(model)
    dt.kv(0, 0, n_max, 0, cache.k, cache.v, **cache.synth_kwargs())
    ref = OracleTrace(model, dt.tabs, 0, n_max, E.EPIKV_SCORE_LAGKV, lag=lag).scores[E.EPIKV_SCORE_LAGKV]
    view = cache.view()
    for n in lengths:
        out = torch.full((n_max + 1,), float("nan"), device="cuda")
        E.epikv_lagkv_score_noalloc(view, 0, n, 2, H, d, lag, 1e-6, 64, out)
        got = out.cpu().numpy()
        assert_scores_close(got[:n], ref[:n], f"n {n}")   # causal: a prefix's scores
        assert np.all(np.isnan(got[n:]))
