"""Evictions of batches up to the 4,096 sequences that a context admits, on the
compaction's routes (equal chunks, per-stream units; per-layer budgets): its
tables in shared memory grow with the batch (a prefix sum per sequence under
token budgets), and 1,536 / 1,537 is where a sequence's outgrow those of the
largest per-layer batch.  Every compacted row is compared with the slot it came
from."""
import pytest
import torch

from paper_2606_26472_gb300 import epikv as E
from paper_2606_26472_gb300.cache import KVCache

pytestmark = pytest.mark.gpu

H, d = 1, 8


def _rows(pool):
    return pool.view(torch.int64).view(*pool.shape[:3], -1)   # [L][S][T][words of a row]


@pytest.mark.parametrize("layers", [0, 1])
@pytest.mark.parametrize("S,T,K,every", [
    (1536, 12, 8, 1), (1537, 12, 8, 1), (4096, 12, 8, 1),
    (4096, 12, 8, 5),       # one entry in five evicts
    (1537, 700, 350, 1),    # shifts beyond the stash, many streams: per-stream units
])
def test_every_sequence_of_a_large_batch(gpu_lib, S, T, K, every, layers):
    L = 2
    cache = KVCache(E.EPIKV_LAYOUT_CONTIGUOUS, L, H, d, max_seqs=S, max_tokens=T)
    g = torch.Generator(device="cuda").manual_seed(5)
    for p in (cache.k, cache.v):
        p.normal_(generator=g)
        p.mul_(torch.exp2(torch.randint(-3, 4, (1, S, T, 1, 1), generator=g, device="cuda").to(p.dtype)))
    cfg = E.make_config(max_seqs=S, max_cache_tokens=T, max_new_tokens=T, num_layers=L, num_kv_heads=H, head_dim=d,
                        lag_window=1, score_kinds=E.EPIKV_SCORE_KVKEY, layer_budgets=layers)
    ws = torch.empty(E.epikv_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    ctx = E.epikv_init(cfg, ws, ws.numel())
    ids = torch.arange(S, dtype=torch.int32, device="cuda").flip(0).contiguous()   # entry b: sequence S - 1 - b
    cu = torch.arange(0, (S + 1) * T, T, dtype=torch.int32, device="cuda")
    for s in range(S):
        E.epikv_seq_reset(ctx, s, 0, E.EPIKV_SCORE_KVKEY)
    E.epikv_score_update(ctx, S, ids, cu, T, None, cache.view())
    before = [_rows(p).clone() for p in (cache.k, cache.v)]
    per = L if layers else 1
    evicts = torch.arange(S, device="cuda") % every == 0
    budget = torch.where(evicts, K, T).to(torch.int32).repeat_interleave(per)
    kept = torch.zeros((S, per, T), dtype=torch.int32, device="cuda")
    n = torch.zeros((S, per), dtype=torch.int32, device="cuda")
    E.epikv_select(ctx, S, ids, budget, None, kept, T, n)
    E.epikv_compact(ctx, S, ids, kept, T, cache.view())
    assert E.epikv_get_error(ctx) == (E.EPIKV_OK, 0)
    assert torch.equal(n.flatten(), budget)
    src = torch.where(evicts[:, None, None], kept, torch.arange(T, dtype=torch.int32, device="cuda")).long()
    slot = torch.arange(T, device="cuda")
    src = torch.where(slot < n[..., None], src, slot)          # slots past the new length are left alone
    src = src.expand(S, L, T).permute(1, 0, 2)[:, ids.long()]  # [layer][sequence][slot] (the ids are their own inverse)
    for p, was in zip((cache.k, cache.v), before):
        want = was.gather(2, src[..., None].expand(-1, -1, -1, was.shape[3]))
        assert torch.equal(_rows(p), want)
    E.epikv_destroy(ctx)
