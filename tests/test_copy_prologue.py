"""The copy kernel's first batches are loaded while the stash kernel, which
zeroes the late chunks' counter, may still run: no CTA's own chunk may end
within them.  Checked on the plan that the kernel follows, at the shipped
thresholds and grids; deeper pipelines that would break it do not compile."""
import pytest

from .plans import compile_plans, plans


@pytest.mark.parametrize("G", [1, 7, 152, 304, 456, 512])
@pytest.mark.parametrize("tails", [False, True])
def test_own_chunks_outlast_the_first_batches(G, tails):
    p = plans()
    least = p.kLateRowsTails if tails else p.kLateRows
    late_seen = False
    for total in (least * G - 1, least * G, least * G + 1, least * G + G - 1, 3 * least * G + 11, 10**9):
        for stride in ([p.kStashRows] if tails else [1, 10, 64, p.kStashRows]):
            for paged in (False, True):
                st = p.chunks(total, G, tails=tails, stride=stride, paged=paged)
                n = len(st) - 1
                assert st[0] == 0 and st[-1] == total and all(a <= b for a, b in zip(st, st[1:]))
                if total < least * G:
                    assert n == G
                if n > G:   # late chunks: taken from the counter
                    late_seen = True
                    assert min(b - a for a, b in zip(st[:G], st[1:G + 1])) > p.kPrologueRows
                    if not tails:   # every chunk's stash lies in the workspace's, its first row's entry too
                        assert n <= p.kMaxChunks and n * stride <= p.kMaxStashCtas * p.kStashRows
    assert late_seen


def test_no_late_chunks_without_their_code():
    p = plans()
    for n_seq, slots, L, G in [(1, 576, 32, 304), (1, 2047, 32, 304), (3, 1216, 32, 304), (1, 100, 1, 304)]:
        if not p.late_possible(n_seq, slots, L, G):
            total = n_seq * slots * 2 * L   # the most rows that can move
            for tails in (False, True):
                assert p.chunks(total, G, tails=tails, stride=1, paged=False) == \
                    p.chunks(total, G, tails=tails, stride=1, paged=False, late=False)
    assert not p.late_possible(1, 576, 32, 304) and p.late_possible(8, 4160, 32, 304)


@pytest.mark.parametrize("stages,ok", [(4, True), (6, True), (7, False), (16, False)])
def test_pipelines_too_deep_for_the_order_do_not_compile(stages, ok):
    r = compile_plans(defines=["EPIKV_COMPACT_STAGES=%d" % stages])
    assert (r.returncode == 0) == ok, r.stderr
    if not ok:
        assert "waited for the stash kernel" in r.stderr
