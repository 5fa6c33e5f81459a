"""The kernels' plans (csrc/plans.h), compiled for the host: what the CPU tests
check is the arithmetic that the kernels run, not a copy of it."""
import ctypes as C
import functools
import os
import shutil
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_26472_gb300", "csrc")

_SOURCE = r"""
#include "plans.h"
using namespace epikv;
extern "C" {
// the chunks' first rows and the end, into `start` ; returns their number
int plan_chunks(int with_late, int stash_rows, int64_t total, int G, int tails, int stride, int paged, int64_t* start) {
  auto fill = [&](auto k) {
    for (int c = 0; c <= k.n; ++c) start[c] = k.start(c);
    return k.n;
  };
  return with_late ? fill(make_chunks<true>(stash_rows, total, G, tails, stride, paged))
                   : fill(make_chunks<false>(stash_rows, total, G, tails, stride, paged));
}
int plan_late_possible(int n_seq, int slots, int L, int G) { return late_possible(n_seq, slots, L, G); }
int plan_stash_stride(int64_t total, int G, int shift, int stash_rows) {
  return chunks_fit_stash(total, G, stash_rows) ? stash_rows : shift_stride(shift, stash_rows);
}
int plan_tail_start(const int32_t* kl, int first, int n_new) {
  return tail_start([kl](int i) { return kl[i]; }, first, n_new);
}
int plan_lag_piece_start(int p0, int lag, int piece, int z) { return lag_piece_start(p0, lag, piece, z); }
int plan_lag_pieces(int max_new, int lag, int piece) { return lag_pieces(max_new, lag, piece); }
int plan_lag_piece_tokens(int L, int lag, int n_seq, int max_new, int num_sms) {
  return lag_piece_tokens(L, lag, n_seq, max_new, num_sms);
}
}
"""
_NAMES = ("kMaxStashCtas", "kStashRows", "kMaxChunks", "kPrologueRows", "kLateRows", "kLateRowsTails", "kLatePerCtaTails")


def compile_plans(out=None, defines=()):
    """g++ over the plans; without `out` their syntax and static assertions only."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        raise RuntimeError("no C++ compiler found for the plans")
    consts = "".join('extern "C" int64_t const_%s() { return epikv::%s; }\n' % (n, n) for n in _NAMES)
    cmd = [cxx, "-std=c++17", "-O1", "-Wall", "-Wno-unknown-pragmas", "-I" + CSRC, *("-D" + d for d in defines), "-x", "c++", "-"]
    cmd += ["-shared", "-fPIC", "-o", out] if out else ["-fsyntax-only"]
    return subprocess.run(cmd, input=_SOURCE + consts, capture_output=True, text=True)


class Plans:
    def __init__(self, path):
        self._lib = C.CDLL(path)
        for n in _NAMES:
            f = getattr(self._lib, "const_" + n)
            f.restype = C.c_int64
            setattr(self, n, f())
        self._lib.plan_chunks.argtypes = [C.c_int, C.c_int, C.c_int64, C.c_int, C.c_int, C.c_int, C.c_int,
                                          C.POINTER(C.c_int64)]
        self.late_possible = self._lib.plan_late_possible
        self.lag_piece_start = self._lib.plan_lag_piece_start
        self.lag_pieces = self._lib.plan_lag_pieces
        self.lag_piece_tokens = self._lib.plan_lag_piece_tokens
        self._lib.plan_stash_stride.argtypes = [C.c_int64, C.c_int, C.c_int, C.c_int]

    def chunks(self, total, G, *, tails, stride, paged, stash_rows=None, late=True):
        """The first row of every chunk, and the end."""
        out = (C.c_int64 * (max(self.kMaxChunks, (self.kLatePerCtaTails + 1) * G) + 1))()
        n = self._lib.plan_chunks(late, self.kStashRows if stash_rows is None else stash_rows, total, G, tails, stride,
                                  paged, out)
        return list(out[:n + 1])

    def stash_stride(self, total, G, shift):
        """Rows of a chunk's stash, 0 if the balanced split does not apply."""
        return self._lib.plan_stash_stride(total, G, shift, self.kStashRows)

    def tail_start(self, kl, first, n_new):
        return self._lib.plan_tail_start((C.c_int32 * len(kl))(*kl), first, n_new)


@functools.lru_cache(None)
def plans():
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "plans.so")
        r = compile_plans(path)
        assert r.returncode == 0, r.stderr
        return Plans(path)
