"""Evictions whose largest shift and chunks exceed the compaction's stash: the
rows whose sources lie below the new length are moved first, in place, the
others in equal chunks.  Deep cuts at several ratios, one sequence and mixed
batches, rows of one vector and of odd widths, both layouts, and a batch of
many streams that keeps one unit per stream; every compacted row is compared
with the slot it came from."""
import numpy as np
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache
from synth import gen

pytestmark = pytest.mark.gpu


def _cut(L, H, d, lengths, budgets, layout, prefill=None, seed=3):
    """Random scores (K/V rows of random amplitude), one eviction of every
    sequence; returns how many kept slots each sequence has."""
    S, T = len(lengths), max(lengths)
    table = None
    if layout == E.EPIKV_LAYOUT_PAGED:
        nb = -(-T // 16)
        table = gen.block_permutation(seed, S * nb).reshape(S, nb)
    cache = KVCache(layout, L, H, d, max_seqs=S, max_tokens=T, block_table=table)
    g = torch.Generator(device="cuda").manual_seed(seed)
    for p in (cache.k, cache.v):
        p.normal_(generator=g)
        p.mul_(torch.exp2(torch.randint(-3, 4, p.shape[:-2], generator=g, device="cuda").to(p.dtype))[..., None, None])
    cfg = E.make_config(max_seqs=S, max_cache_tokens=T, max_new_tokens=T, num_layers=L, num_kv_heads=H, head_dim=d,
                        lag_window=1, score_kinds=E.EPIKV_SCORE_KVKEY)
    ws = torch.empty(E.epikv_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    ctx = E.epikv_init(cfg, ws, ws.numel())
    ids = torch.arange(S, dtype=torch.int32, device="cuda")
    cu = torch.tensor([0] + list(np.cumsum(lengths)), dtype=torch.int32, device="cuda")
    for s in range(S):
        E.epikv_seq_reset(ctx, s, prefill[s] if prefill else 0, E.EPIKV_SCORE_KVKEY)
    E.epikv_score_update(ctx, S, ids, cu, T, None, cache.view())
    before = [[cache.rows(kv, s, np.arange(lengths[s])).clone() for kv in range(2)] for s in range(S)]
    stride = max(max(budgets), max(prefill or [0]))
    kept = torch.zeros((S, stride), dtype=torch.int32, device="cuda")
    n = torch.zeros(S, dtype=torch.int32, device="cuda")
    E.epikv_select(ctx, S, ids, torch.tensor(budgets, dtype=torch.int32, device="cuda"), None, kept, stride, n)
    E.epikv_compact(ctx, S, ids, kept, stride, cache.view())
    E.epikv_compact(ctx, S, ids, kept, stride, cache.view())   # applied once: moves nothing
    assert E.epikv_get_error(ctx) == (E.EPIKV_OK, 0)
    counts = n.tolist()
    for s in range(S):
        src = kept[s, :counts[s]].long() if counts[s] < lengths[s] else torch.arange(lengths[s], device="cuda")
        tail = np.arange(counts[s], lengths[s])   # slots past the new length are left alone
        for kv in range(2):
            after = cache.rows(kv, s, np.arange(counts[s]))
            assert torch.equal(after.view(torch.int16), before[s][kv].index_select(0, src).view(torch.int16)), (s, kv)
            assert torch.equal(cache.rows(kv, s, tail).view(torch.int16), before[s][kv][counts[s]:].view(torch.int16))
    E.epikv_destroy(ctx)
    return counts


@pytest.mark.parametrize("layout", [E.EPIKV_LAYOUT_PAGED, E.EPIKV_LAYOUT_CONTIGUOUS])
@pytest.mark.parametrize("L,H,d,lengths,budgets,prefill", [
    (32, 8, 128, (6000,), (2000,), None),                     # a third kept
    (32, 8, 128, (9001,), (1500,), None),                     # a sixth
    (32, 8, 128, (4000,), (3600,), None),                     # nearly all: almost every row is in the head
    (16, 8, 128, (9000, 4000, 700, 5000), (1300, 1999, 800, 4700), (0, 300, 0, 7)),   # mixed, one untouched
    (64, 1, 8, (8000, 8000), (2500, 4000), None),             # rows of one vector
    (32, 3, 8, (9000,), (3000,), (2900,)),                    # rows of three vectors; hardly a candidate
    (24, 5, 64, (7000, 300), (3000, 290), None),              # rows of 40 vectors, and a shift within the stash
    (48, 8, 256, (4500,), (2047,), None),                     # the widest rows
])
def test_deep_cuts(gpu_lib, L, H, d, lengths, budgets, prefill, layout):
    counts = _cut(L, H, d, lengths, budgets, layout, prefill)
    assert counts == [min(n, max(k, (prefill or [0] * 9)[i])) for i, (n, k) in enumerate(zip(lengths, budgets))]


def test_many_streams_keep_their_units(gpu_lib):
    """24 sequences x 64 streams, 600 -> 300 slots: heads of half the rows and
    five streams per CTA."""
    assert _cut(32, 1, 64, (600,) * 24, (300,) * 24, E.EPIKV_LAYOUT_CONTIGUOUS) == [300] * 24


@pytest.mark.parametrize("L,lengths,budgets,layout", [
    (32, (10200,), (10072,), E.EPIKV_LAYOUT_PAGED),             # shift 128: as many chunks as the whole stash holds
    (32, (10200,), (10190,), E.EPIKV_LAYOUT_CONTIGUOUS),        # shift 10
    (64, (5100, 3000, 90, 2500), (5040, 2999, 100, 2440), E.EPIKV_LAYOUT_CONTIGUOUS),
    (64, (5200, 5150), (5100, 5149), E.EPIKV_LAYOUT_PAGED),
])
def test_long_copies_with_late_chunks(gpu_lib, L, lengths, budgets, layout):
    """More than 2,048 moved rows per CTA: the shorter chunks at the end of the
    row space, taken as the CTAs finish, and their stashes of the largest
    shift's rows."""
    assert _cut(L, 1, 64, lengths, budgets, layout, prefill=(3,) * len(lengths)) == [min(a, b) for a, b in
                                                                                     zip(lengths, budgets)]
