"""The bytes that the bench credits to a deep cut's two moving kernels: the rows
that each of them moves, by the kernels' own rule (rows from the first one whose
source lies at or past the new length are the tail), and together every moved row."""
import numpy as np
import pytest


@pytest.mark.parametrize("n,K,seed", [(65536, 4096, 1), (4396, 4096, 2), (700, 699, 3), (40, 1, 4), (12, 12, 5)])
def test_each_kernel_is_credited_with_its_own_rows(n, K, seed):
    import bench
    rng = np.random.default_rng(seed)
    kept = np.stack([np.sort(rng.choice(n, K, replace=False)) for _ in range(3)])
    rows = {"compact_stash_kernel": 0, "compact_kernel": 0}
    for kl in kept:
        first = next((i for i in range(K) if kl[i] != i), K)
        tail = next((i for i in range(first, K) if kl[i] >= K), K)
        rows["compact_stash_kernel"] += tail - first
        rows["compact_kernel"] += K - tail
    assert bench.deep_cut_bytes(kept, 1000) == {k: 2 * r * 1000 for k, r in rows.items()}
    if n > 10 * K > 10:   # a deep cut: the heads are few, and the copy is not credited with them
        t = bench.kernel_table([("_ZN5epikv14compact_kernelEv", 1.0), ("_ZN5epikv20compact_stash_kernelEv", 0.1)], 1,
                               bench.deep_cut_bytes(kept, 1000), 6000.0)
        assert t["compact_kernel"]["gbs"] == pytest.approx(2 * rows["compact_kernel"] * 1000 / 1e6)
        assert t["compact_stash_kernel"]["gbs"] == pytest.approx(2 * rows["compact_stash_kernel"] * 1000 / 1e5)
