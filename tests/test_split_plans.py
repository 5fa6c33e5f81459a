"""The plans of the split kernels (csrc/plans.h, compiled for the host) checked
by brute force on the CPU: the chunks of the compaction's balanced split at the
shipped thresholds (one per CTA and, for long copies, shorter late ones, copied
in any order), the head and tail split of deep cuts with its search, and the
pieces of long K/V score updates.  What the kernels do with a plan (which
sources are stashed, a batch's loads before its stores) is restated here; the
GPU tests compare its results."""
import random

import pytest

from .plans import plans


def kept_list(rng, n, k, spread=None):
    """A random ascending kept list of k of n slots; with `spread`, the evicted
    ones lie among the first slots only."""
    ev = set(rng.sample(range(spread or n), n - k))
    return [i for i in range(n) if i not in ev]


@pytest.mark.parametrize("late", [False, True])
@pytest.mark.parametrize("seed", range(12))
def test_chunks_in_any_order_leave_every_row_in_place(seed, late):
    p, rng = plans(), random.Random(2 * seed + late)
    G = rng.choice([1, 2, 3] if late else [3, 20, 304])
    per_cta = rng.choice([p.kLateRows, p.kLateRows + 1, 2500] if late else [5, 100, 400, p.kLateRows - 40])
    max_shift = rng.choice([1, 9, p.kStashRows, 300])
    streams, n_rows = [], 0   # (kept, first, n_new, n), several streams of each entry
    while n_rows < per_cta * G:
        n = rng.randint(400, 1500)
        kl = kept_list(rng, n, n - rng.randint(1, max_shift))
        first = next((i for i, s in enumerate(kl) if s != i), len(kl))
        if first < len(kl):
            streams += [(kl, first, len(kl), n)] * rng.randint(1, 4)
            n_rows = sum(s[2] - s[1] for s in streams)
    rows = [(s, i) for s, (kl, first, n_new, n) in enumerate(streams) for i in range(first, n_new)]
    shift = max(kl[-1] - (len(kl) - 1) for kl, *_ in streams)
    stride = p.stash_stride(len(rows), G, shift)
    if stride == 0:
        assert shift > p.kStashRows and -(-len(rows) // G) > p.kStashRows
        return
    assert stride <= p.kStashRows
    paged = rng.random() < 0.5
    st = p.chunks(len(rows), G, tails=False, stride=stride, paged=paged)
    n = len(st) - 1
    assert st[0] == 0 and st[-1] == len(rows) and all(a <= b for a, b in zip(st, st[1:]))
    assert n == G if not late and len(rows) < p.kLateRows * G else n > G
    assert n <= p.kMaxChunks and n * stride <= p.kMaxStashCtas * p.kStashRows
    cache = [list(range(n)) for *_, n in streams]
    stash = {}
    for g in range(1, n):   # the sources of the chunk before, in the region from row a on
        if st[g] >= len(rows):
            continue
        s, a = rows[st[g]]
        kl, first, n_new, _ = streams[s]
        if a == first:
            continue
        x = [i for i in range(max(first, a - (st[g] - st[g - 1])), a) if a <= kl[i] < n_new]
        assert len(x) <= stride and (not x or x == list(range(x[0], x[-1] + 1)))   # a run within the stash
        stash[g] = {kl[i]: cache[s][kl[i]] for i in x}
    order = list(range(n))
    rng.shuffle(order)
    for g in order:
        o = st[g]
        while o < st[g + 1]:
            s, i = rows[o]
            kl, first, n_new, _ = streams[s]
            end = min(n_new, i + st[g + 1] - o)   # the chunk's rows of this stream; another chunk's follow if end < n_new
            for r in range(i, end):
                cache[s][r] = stash[g + 1][kl[r]] if end < n_new and end <= kl[r] < n_new else cache[s][kl[r]]
            o += end - i
    for (kl, first, n_new, n), c in zip(streams, cache):
        assert c[:n_new] == kl and c[n_new:] == list(range(n_new, n))


@pytest.mark.parametrize("seed", range(60))
def test_heads_then_tails_leave_every_row_in_place(seed):
    rng = random.Random(1000 + seed)
    n = rng.randint(2, 900)
    k = rng.randint(1, n - 1)
    kl = kept_list(rng, n, k, spread=rng.choice([None, max(n - k, n // 2)]))
    n_new = len(kl)
    first = next((i for i, s in enumerate(kl) if s != i), n_new)
    cut = plans().tail_start(kl, first, n_new)
    assert cut == first + sum(s < n_new for s in kl[first:])
    cache = list(range(n))
    batch = rng.choice([1, 7, 64])
    for i0 in range(first, cut, batch):   # the head: a batch's loads before its stores
        take = [cache[kl[i]] for i in range(i0, min(cut, i0 + batch))]
        cache[i0:i0 + len(take)] = take
    tail = list(range(cut, n_new))
    rng.shuffle(tail)                     # the tail: in any order
    for i in tail:
        cache[i] = cache[kl[i]]
    assert cache[:n_new] == kl and cache[n_new:] == list(range(n_new, n))


def _check_pieces(p0, lag, piece, max_new, lengths):
    p = plans()
    z_n = p.lag_pieces(max_new, lag, piece)
    start = [p.lag_piece_start(p0, lag, piece, z) for z in range(z_n + 1)]
    for n_new in lengths:
        taken = []
        for z in range(z_n):
            lo, hi = start[z], min(n_new, start[z + 1])
            if lo >= n_new and z > 0:
                continue
            taken += range(lo, hi)
            if z > 0:
                assert (p0 + lo) % lag == 0 and lo - lag >= 0    # the chunk before the cut is the call's
        assert taken == list(range(n_new))
        if n_new > start[1]:   # the first piece writes the state from the call's own rows
            tail = (p0 + n_new) % lag
            assert n_new - tail - lag >= 0


@pytest.mark.parametrize("seed", range(60))
def test_pieces_cover_a_call_and_cut_at_chunks(seed):
    rng = random.Random(2000 + seed)
    lag = rng.choice([1, 2, 7, 16, 100])
    piece = lag * rng.randint(4, 20)
    p0, max_new = rng.randint(0, 5 * lag), rng.randint(1, 40 * piece // lag + 3 * piece)
    _check_pieces(p0, lag, piece, max_new, {max_new, rng.randint(0, max_new)})


@pytest.mark.parametrize("seed", range(60))
def test_pieces_that_calls_are_cut_into(seed):
    rng = random.Random(3000 + seed)
    lag, L, n_seq = rng.choice([1, 3, 7, 16, 100, 5000]), rng.choice([1, 2, 32, 80]), rng.choice([1, 2, 9, 200])
    max_new = int(2 ** rng.uniform(0, 16))
    piece = plans().lag_piece_tokens(L, lag, n_seq, max_new, 152)
    if piece == 0:
        assert plans().lag_pieces(max_new, lag, piece) == 1
        return
    assert piece % lag == 0 and 4 * lag <= piece < max_new and max_new >= 128
    assert plans().lag_pieces(max_new, lag, piece) <= 65535   # grid.z
    _check_pieces(rng.randint(0, 3 * lag), lag, piece, max_new, {max_new, 1, rng.randint(0, max_new)})
