"""Per-layer budgets with a copy long enough for late chunks, cut within the
stash (balanced split) and beyond it (units taken from the shared counter),
several steps in a row from one context: every layer's compacted rows are the
rows of the positions that the layer holds."""
import numpy as np
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("new", [60, 400])
def test_layer_rows_over_steps(gpu_lib, new):
    L, H, d, S = 64, 1, 64, 2
    base = 6000
    budgets = [base - 20 * l for l in range(L)]
    T = base + new
    cache = KVCache(E.EPIKV_LAYOUT_CONTIGUOUS, L, H, d, max_seqs=S, max_tokens=T)
    cfg = E.make_config(max_seqs=S, max_cache_tokens=T, max_new_tokens=T, num_layers=L, num_kv_heads=H, head_dim=d,
                        lag_window=1, score_kinds=E.EPIKV_SCORE_KVKEY, layer_budgets=1)
    ws = torch.empty(E.epikv_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    ctx = E.epikv_init(cfg, ws, ws.numel())
    ids = torch.arange(S, dtype=torch.int32, device="cuda")
    bud = torch.tensor(budgets * S, dtype=torch.int32, device="cuda")
    for s in range(S):
        E.epikv_seq_reset(ctx, s, 0, E.EPIKV_SCORE_KVKEY)
    gen = torch.Generator(device="cuda").manual_seed(7)
    held = np.zeros((S, L), dtype=int)
    rows = {}       # (sequence, layer): the rows its slots hold, by position

    def step(n):
        for s in range(S):
            amp = torch.exp2(torch.randint(-3, 4, (n, 1, 1), generator=gen, device="cuda").float())
            for l in range(L):
                x = [(torch.randn((n, H, d), generator=gen, device="cuda") * amp).to(torch.bfloat16) for _ in range(2)]
                for kv in range(2):
                    cache.write_layer_rows(kv, s, l, np.arange(held[s, l], held[s, l] + n), x[kv])
                old = rows.get((s, l))
                rows[s, l] = x if old is None else [torch.cat([a, b]) for a, b in zip(old, x)]
        cu = torch.tensor([n * i for i in range(S + 1)], dtype=torch.int32, device="cuda")
        E.epikv_step(ctx, S, ids, cu, n, bud, None, None, cache.view())
        assert E.epikv_get_error(ctx) == (E.EPIKV_OK, 0)
        for s in range(S):
            for l in range(L):
                pos, m = E.epikv_read_layer_slots(ctx, s, l, T)
                held[s, l] = m
                for kv, pool in ((0, cache.k), (1, cache.v)):
                    want = rows[s, l][kv].index_select(0, torch.as_tensor(pos, device="cuda"))
                    assert torch.equal(pool[l, s, :m].view(torch.int16), want.view(torch.int16)), (s, l, kv)

    step(base)
    for _ in range(3):
        step(new)
    assert (held == np.array(budgets)).all()
    E.epikv_destroy(ctx)
