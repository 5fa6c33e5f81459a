"""Long score updates whose K/V streams are cut into pieces: bit for bit the
scores, and the state left behind, of the same tokens in short calls (one
piece each), at lags that do not divide anything, odd lengths, ragged batches
and both layouts; and unmapped rows reported whichever piece holds them."""
import numpy as np
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache

pytestmark = pytest.mark.gpu

KV = E.EPIKV_SCORE_LAGKV | E.EPIKV_SCORE_KVKEY | E.EPIKV_SCORE_KVVAL | E.EPIKV_SCORE_LAGKEY


def _ctx(L, H, d, S, T, max_new, lag, kinds):
    cfg = E.make_config(max_seqs=S, max_cache_tokens=T, max_new_tokens=max_new, num_layers=L, num_kv_heads=H, head_dim=d,
                        lag=lag, score_kinds=kinds)
    n = E.epikv_workspace_bytes(cfg)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    ctx = E.epikv_init(cfg, ws, n)
    for s in range(S):
        E.epikv_seq_reset(ctx, s, 0, kinds & -kinds)
    return ctx, ws


def _update(ctx, counts, kv):
    cu = torch.tensor([0] + list(np.cumsum(counts)), dtype=torch.int32, device="cuda")
    ids = torch.arange(len(counts), dtype=torch.int32, device="cuda")
    E.epikv_score_update(ctx, len(counts), ids, cu, max(counts), None, kv)


@pytest.mark.parametrize("L,H,d,lag,lengths,before,layout,kinds", [
    (2, 8, 128, 16, (1201,), 0, E.EPIKV_LAYOUT_PAGED, E.EPIKV_SCORE_LAGKV),
    (2, 8, 128, 16, (1024, 255, 256, 257), 5, E.EPIKV_LAYOUT_CONTIGUOUS, KV),
    (1, 2, 32, 7, (2000, 1, 613), 33, E.EPIKV_LAYOUT_PAGED, E.EPIKV_SCORE_LAGKV | E.EPIKV_SCORE_LAGKEY),
    (3, 1, 8, 1, (777, 300), 2, E.EPIKV_LAYOUT_CONTIGUOUS, KV),
    (1, 4, 64, 100, (2400, 1600), 150, E.EPIKV_LAYOUT_PAGED, E.EPIKV_SCORE_LAGKV),
    (1, 4, 64, 16, (900, 640), 17, E.EPIKV_LAYOUT_CONTIGUOUS, E.EPIKV_SCORE_KVKEY | E.EPIKV_SCORE_KVVAL),
    (32, 1, 32, 16, (600, 533, 600, 257), 3, E.EPIKV_LAYOUT_PAGED, E.EPIKV_SCORE_LAGKV),   # pieces of full length
    (1, 8, 256, 16, (513,), 0, E.EPIKV_LAYOUT_CONTIGUOUS, E.EPIKV_SCORE_LAGKV),
    (2, 8, 128, 600, (1300,), 0, E.EPIKV_LAYOUT_CONTIGUOUS, E.EPIKV_SCORE_LAGKV),   # no cut: pieces shorter than 8 chunks
])
def test_pieces_equal_short_calls(L, H, d, lag, lengths, before, layout, kinds):
    S, after = len(lengths), 40
    T = max(lengths) + before + after
    kvc = KVCache(layout, L, H, d, max_seqs=S, max_tokens=T)
    gen = torch.Generator(device="cuda").manual_seed(11)
    for p in (kvc.k, kvc.v):
        p.normal_(generator=gen)
    kv = kvc.view()
    scores = []
    for step in (max(lengths), 61):   # 61 < two pieces: never cut
        ctx, ws = _ctx(L, H, d, S, T, max(max(lengths), before, after, 1), lag, kinds)
        if before:
            for at in range(0, before, 61):
                _update(ctx, [min(61, before - at)] * S, kv)
        for at in range(0, max(lengths), step):
            _update(ctx, [max(0, min(step, n - at)) for n in lengths], kv)
        _update(ctx, [after] * S, kv)   # scored from the state the long call left
        assert E.epikv_get_error(ctx) == (E.EPIKV_OK, 0)
        got = {}
        for s in range(S):
            for k in range(6):
                if kinds >> k & 1:
                    pos, sc, n = E.epikv_read_slots(ctx, s, 1 << k, T)
                    assert n == before + lengths[s] + after
                    got[s, k] = np.array(sc, np.float32).view(np.uint32)
        scores.append(got)
        E.epikv_destroy(ctx)
    for key in scores[0]:
        np.testing.assert_array_equal(scores[0][key], scores[1][key], err_msg=str(key))


def test_unmapped_row_in_a_later_piece_is_reported():
    kvc = KVCache(E.EPIKV_LAYOUT_PAGED, 1, 2, 32, max_seqs=1, max_tokens=1024)
    kvc.k.normal_()
    kvc.v.normal_()
    bt = kvc.block_table.clone()
    bt[0, 700 // 16] = -1
    ctx, ws = _ctx(1, 2, 32, 1, 1024, 1024, 16, E.EPIKV_SCORE_LAGKV)
    _update(ctx, [1000], kvc.view(bt))
    assert E.epikv_get_error(ctx) == (E.EPIKV_EDEVICE, E.EPIKV_DEV_SLOT)
    E.epikv_destroy(ctx)
