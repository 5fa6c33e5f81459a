"""The plans of the split kernels, restated and checked by brute force on the
CPU: the chunks of long copies (one per CTA and shorter late ones, in any
order), the head and tail split of deep cuts with its search, and the pieces
of long K/V score updates."""
import random

import pytest

KMAX_STASH_CTAS, KMAX_CHUNKS, KCHUNKS_PAGED = 512, 1024, 768


def chunk_starts(total, G, tails, stride, paged, stash_rows, late_rows, late_rows_tails):
    """Chunks::start of csrc/compact.cu for every chunk, and the end."""
    late = 0
    if tails:
        late = 8 * G if total >= late_rows_tails * G else 0
    elif total >= late_rows * G:
        late = min(min(KCHUNKS_PAGED if paged else KMAX_CHUNKS, KMAX_STASH_CTAS * stash_rows // stride) - G, 3 * G)
    late = max(late, 0)
    early = total - total * late // G * (20 if tails or paged else 50) // 1000 if late else total
    n = G + late
    return [early * c // G if c <= G else early + (total - early) * (c - G) // (n - G) for c in range(n + 1)]


def kept_list(rng, n, k, spread=None):
    """A random ascending kept list of k of n slots; with `spread`, the evicted
    ones lie among the first slots only."""
    ev = set(rng.sample(range(spread or n), n - k))
    return [i for i in range(n) if i not in ev]


def tail_start(kl, first, n_new):
    """The eight-way search of csrc/compact.cu."""
    lo, hi = first, n_new
    while lo < hi:
        step = (hi - lo + 7) // 8
        below = sum(kl[min(lo + j * step, hi - 1)] < n_new for j in range(8))
        if below == 0:
            return lo
        last = min(lo + (below - 1) * step, hi - 1)
        if below < 8:
            hi = min(lo + below * step, hi - 1)
        lo = last + 1
    return lo


@pytest.mark.parametrize("seed", range(40))
def test_chunks_in_any_order_leave_every_row_in_place(seed):
    rng = random.Random(seed)
    G, stash_rows = rng.choice([3, 8, 20]), 32
    streams = []   # (kept, first, n_new): several streams of a few entries
    for _ in range(rng.randint(1, 3)):
        n = rng.randint(60, 400)
        kl = kept_list(rng, n, n - rng.randint(1, stash_rows))
        first = next(i for i, s in enumerate(kl) if s != i) if kl[-1] != len(kl) - 1 else len(kl)
        if first < len(kl):
            streams += [(kl, first, len(kl), n)] * rng.randint(1, 4)
    rows = [(s, i) for s, (kl, first, n_new, n) in enumerate(streams) for i in range(first, n_new)]
    chunk_of = {}
    shift = max((kl[-1] - (len(kl) - 1) for kl, *_ in streams), default=1)
    st = chunk_starts(len(rows), G, False, shift, rng.random() < 0.5, stash_rows, 2, 2)
    assert st[0] == 0 and st[-1] == len(rows) and all(a <= b for a, b in zip(st, st[1:]))
    assert (len(st) - 1) * shift <= KMAX_STASH_CTAS * stash_rows or len(st) - 1 == G
    for g in range(len(st) - 1):
        chunk_of.update((x, g) for x in rows[st[g]:st[g + 1]])
    cache = [list(range(n)) for *_, n in streams]
    stash = {}
    for g in range(1, len(st) - 1):   # the sources of the chunk before, in the region from row a on
        if st[g] >= len(rows):
            continue
        s, a = rows[st[g]]
        kl, first, n_new, _ = streams[s]
        if a == first:
            continue
        start = max(first, a - (st[g] - st[g - 1]))
        x = [i for i in range(start, a) if a <= kl[i] < n_new]
        assert len(x) <= shift and x == list(range(x[0], x[-1] + 1)) if x else True   # a run within the stash
        stash[g] = {kl[i]: cache[s][kl[i]] for i in x}
    order = list(range(len(st) - 1))
    rng.shuffle(order)
    for g in order:
        for s, i in rows[st[g]:st[g + 1]]:
            kl, first, n_new, _ = streams[s]
            end = next((e for e in range(i + 1, n_new) if chunk_of[s, e] != g), n_new)
            stashed = end < n_new and end <= kl[i] < n_new
            cache[s][i] = stash[g + 1][kl[i]] if stashed else cache[s][kl[i]]
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
    cut = tail_start(kl, first, n_new)
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


@pytest.mark.parametrize("seed", range(60))
def test_pieces_cover_a_call_and_cut_at_chunks(seed):
    rng = random.Random(2000 + seed)
    lag = rng.choice([1, 2, 7, 16, 100])
    piece = lag * rng.randint(4, 20)
    p0, max_new = rng.randint(0, 5 * lag), rng.randint(1, 40 * piece // lag + 3 * piece)
    z_n = (max_new + 2 * lag + piece - 1) // piece
    start = [0 if z == 0 else (lag - p0 % lag) % lag + z * piece - 2 * lag for z in range(z_n + 1)]
    for n_new in {max_new, rng.randint(0, max_new)}:
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
