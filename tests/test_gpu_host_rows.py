"""lx_lex_host on the row kernels (csrc/rows.cu: lex_rows_host) against the
oracle, element by element: one piece and several, sizes at the edge where a
second piece starts, an error in the first, a middle and the last piece, a
capacity that ends inside a piece, and pieces that the row kernels hand over
(lookahead that fails across more than they follow)."""

import numpy as np
import pytest

import oracle
from lexinputs import corpus
from lexinputs import tokensets as T

pytestmark = pytest.mark.gpu
PIECE = 12 << 20   # csrc/lex.cu: ROWS_PIECE


@pytest.fixture(scope="module")
def env(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib, lexlib.lx_ctx_create()


def check(lg, ctx, name, w, mode, cap=None, pin=True):
    import torch
    dfa, disc = T.tokenset(name), T.discarded_kinds(name)
    ts = lg.lx_compile_tokenset(dfa, disc)
    ek, el, econ = oracle.lex(dfa, w)
    if mode:
        ek, el = oracle.discard(ek, el, disc, dfa.n_kinds)
    cap = ek.size if cap is None else cap
    h = torch.from_numpy(np.ascontiguousarray(w).copy())
    k = torch.full((cap + 8,), -1, dtype=torch.int16)
    l = torch.full((cap + 8,), -1, dtype=torch.int32)
    if pin:
        h, k, l = h.pin_memory(), k.pin_memory(), l.pin_memory()
    rc, nt, con = lg.lx_lex_host(ctx, ts, h, mode, k, l, capacity=cap)
    assert rc == (0 if ek.size <= cap else lg.LX_E_CAPACITY), lg.lx_strerror(rc)
    assert (nt, con) == (ek.size, econ)
    m = min(nt, cap)
    assert np.array_equal(k[:m].numpy().view(np.uint16).astype(np.int64), ek[:m])
    assert np.array_equal(l[:m].numpy().view(np.uint32).astype(np.int64), el[:m])
    assert (k[cap:] == -1).all() and (l[cap:] == -1).all()


@pytest.mark.parametrize("n", [1, 31, 4096, (4 << 20) + 1, 2 * PIECE - 1, 2 * PIECE + 7, 3 * PIECE + 5])
@pytest.mark.parametrize("name,mode", [("json", 2), ("clike", 0)])
def test_sizes(env, name, mode, n):
    lg, ctx = env
    check(lg, ctx, name, corpus.generate(name, n, seed=321), mode, pin=n % 2 == 1)


def test_errors_and_capacity(env):
    lg, ctx = env
    n = 3 * PIECE + 5
    w = corpus.generate("json", n, seed=322)
    for pos in (0, PIECE // 2, PIECE, n // 2, n - 1):
        bad = w.copy()
        bad[pos] = 1
        check(lg, ctx, "json", bad, 2)
    for cap in (0, 1, 1_000_003):
        check(lg, ctx, "json", w, 2, cap=cap)


def test_pieces_handed_over(env):
    # over a, a+b and ; : an a that no b follows is found by lookahead to the next ';'
    lg, ctx = env
    base = np.frombuffer(b"aab;ab;;" * (2 * PIECE // 8 + 100), np.uint8)
    check(lg, ctx, "lookahead", base, 0)
    for at in (1000, base.size - 3000):
        w = base.copy()
        w[at:at + 900] = ord("a")
        w[at + 900] = ord(";")
        check(lg, ctx, "lookahead", w, 0)
