"""Per-layer budgets at the edge of the selection's staging: caches of up to
24,576 slots have their keys and bits in shared memory, longer ones are read in
every pass.  Distinct and much repeated scores (repeated: which of the slots
equal to the threshold are kept matters); every layer's positions equal the
oracle's replay on the GPU's own scores, and its compacted rows are the rows of
those positions."""
import numpy as np
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache

from .harness import LayerReplay

pytestmark = pytest.mark.gpu

L, H, d, S, NEW, STEPS = 3, 1, 8, 2, 600, 3


@pytest.mark.parametrize("repeated", [False, True])
@pytest.mark.parametrize("T", [24576, 24577, 40003])
def test_long_caches_at_both_routes(gpu_lib, T, repeated):
    budgets, prefill = [T - NEW - 900 * l for l in range(L)], (0, 9)
    cache = KVCache(E.EPIKV_LAYOUT_CONTIGUOUS, L, H, d, max_seqs=S, max_tokens=T)
    cfg = E.make_config(max_seqs=S, max_cache_tokens=T, max_new_tokens=T, num_layers=L, num_kv_heads=H, head_dim=d,
                        lag_window=1, score_kinds=E.EPIKV_SCORE_KVKEY, layer_budgets=1)
    ws = torch.empty(E.epikv_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    ctx = E.epikv_init(cfg, ws, ws.numel())
    ids = torch.arange(S, dtype=torch.int32, device="cuda")
    bud = torch.tensor(budgets * S, dtype=torch.int32, device="cuda")
    kept = torch.zeros((S, L, T), dtype=torch.int32, device="cuda")
    n_kept = torch.zeros((S, L), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(T + repeated)
    total = T + STEPS * NEW
    # every position's rows [K|V][sequence][layer][position]; repeated: the keys are one of 40 in all layers
    rows = torch.randn((2, S, L, total, H, d), generator=gen, device="cuda")
    rows *= torch.exp2(torch.randint(-3, 4, (2, S, L, total, 1, 1), generator=gen, device="cuda").float())
    if repeated:
        rows[0] = rows[0, :, :1, :40].expand(S, L, 40, H, d)[:, :, torch.randint(40, (total,), generator=gen, device="cuda")]
    rows = rows.to(torch.bfloat16)
    replay = [LayerReplay(L, budgets, prefill[s], max(budgets)) for s in range(S)]
    for s in range(S):
        E.epikv_seq_reset(ctx, s, prefill[s], E.EPIKV_SCORE_KVKEY)
    held, seen = np.zeros((S, L), dtype=int), 0
    for n in [T] + [NEW] * STEPS:
        for s in range(S):
            for l in range(L):
                for kv in range(2):
                    cache.write_layer_rows(kv, s, l, np.arange(held[s, l], held[s, l] + n), rows[kv, s, l, seen:seen + n])
        cu = torch.tensor([n * i for i in range(S + 1)], dtype=torch.int32, device="cuda")
        E.epikv_score_update(ctx, S, ids, cu, n, None, cache.view())
        for s in range(S):
            pos, sc, m = E.epikv_read_slots(ctx, s, E.EPIKV_SCORE_KVKEY, T)
            replay[s].append(pos[m - n:], sc[m - n:])
            if repeated and n == T:
                assert len(np.unique(sc)) <= 40
        seen += n
        E.epikv_select(ctx, S, ids, bud, None, kept, T, n_kept)
        E.epikv_compact(ctx, S, ids, kept, T, cache.view())
        assert E.epikv_get_error(ctx) == (E.EPIKV_OK, 0)
        for s in range(S):
            assert replay[s].event()
            for l in range(L):
                pos, held[s, l] = E.epikv_read_layer_slots(ctx, s, l, T)
                np.testing.assert_array_equal(pos, replay[s].caches[l])
                at = torch.as_tensor(np.array(pos), device="cuda").long()
                for kv, pool in ((0, cache.k), (1, cache.v)):
                    assert torch.equal(pool[l, s, :held[s, l]].view(torch.int16), rows[kv, s, l, at].view(torch.int16))
        assert n_kept.tolist() == held.tolist() == [budgets] * S
    E.epikv_destroy(ctx)
