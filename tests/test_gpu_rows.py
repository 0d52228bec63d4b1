"""lx_lex from entry rows (csrc/rows.cu) against the oracle, element by
element: sizes at the edges of blocks, slices, tiles and of the range in which
one kernel finds the rows and lexes, every input alignment, tokens longer than
a stage entry's length field, a slice and a tile, lexing errors and
backtracking at slice edges (some of which the call hands to the other
paths), capacities that cut a tile, and random automata."""

import random

import numpy as np
import pytest

import oracle
from lexinputs import corpus
from lexinputs import tokensets as T

from test_oracle_bruteforce import _random_automata

pytestmark = pytest.mark.gpu
FUSED = 4 << 20   # csrc/rows.cu: FUSED_MAX


@pytest.fixture(scope="module")
def env(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib, lexlib.lx_ctx_create()


_ts = {}


def compiled(lg, name):
    if name not in _ts:
        _ts[name] = lg.lx_compile_tokenset(T.tokenset(name), T.discarded_kinds(name))
    return _ts[name]


def check(lg, ctx, ts, dfa, disc, w, mode, off=0, cap=None):
    import torch
    w = np.frombuffer(bytes(w), np.uint8) if isinstance(w, (bytes, bytearray)) else np.ascontiguousarray(w)
    n = int(w.size)
    buf = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")
    d = buf[off:off + n]
    d.copy_(torch.from_numpy(w.copy()))
    full = n + 1 if cap is None else cap
    k = torch.full((full + 8,), -1, dtype=torch.int16, device="cuda")
    l = torch.full((full + 8,), -1, dtype=torch.int32, device="cuda")
    rc, nt, con = lg.lx_lex(ctx, ts, d, mode, k, l, n=n, capacity=full)
    ek, el, econ = oracle.lex(dfa, w)
    if mode:
        ek, el = oracle.discard(ek, el, disc, dfa.n_kinds)
    assert rc == (0 if ek.size <= full else lg.LX_E_CAPACITY), lg.lx_strerror(rc)
    assert (nt, con) == (ek.size, econ)
    m = min(nt, full)
    assert np.array_equal(k[:m].cpu().numpy().view(np.uint16).astype(np.int64), ek[:m])
    assert np.array_equal(l[:m].cpu().numpy().view(np.uint32).astype(np.int64), el[:m])
    assert (k[full:] == -1).all() and (l[full:] == -1).all()   # nothing past the capacity


@pytest.mark.parametrize("name,mode", [("json", 2), ("json", 0), ("clike", 2), ("arith", 0)])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 1023, 1024, 1025, 2049, 40000, FUSED - 1, FUSED, FUSED + 1,
                               5 * (1 << 20) + 7])
def test_sizes_and_alignment(env, name, mode, n):
    lg, ctx = env
    dfa, disc = T.tokenset(name), T.discarded_kinds(name)
    w = corpus.generate(name, n, seed=300 + n % 97)
    for off in ((0, 1, 15) if n < 50000 else (0, 13)):
        check(lg, ctx, compiled(lg, name), dfa, disc, w, mode, off=off)


@pytest.mark.parametrize("total", [60_000, FUSED + 300_000])
def test_long_tokens(env, total):
    lg, ctx = env
    dfa, disc = T.tokenset("json"), T.discarded_kinds("json")
    base = corpus.generate("json", total, seed=311)
    nl = np.flatnonzero(base == 10)
    parts, at = [], 0
    for i, length in enumerate([509, 510, 511, 512, 513, 1024, 2049, 6143, 6144, 7000, 20000]):
        cut = int(nl[(i + 1) * nl.size // 14]) + 1
        parts += [base[at:cut].tobytes(), b'"' + b"z" * (length - 2) + b'"\n', b" " * length]
        at = cut
    w = b"".join(parts) + base[at:].tobytes()
    for mode in (0, 1, 2):
        check(lg, ctx, compiled(lg, "json"), dfa, disc, w, mode)


@pytest.mark.parametrize("total", [50_000, FUSED + 100_000])
def test_errors_at_slice_edges(env, total):
    lg, ctx = env
    rng = random.Random(5)
    for name, mode, bad in (("json", 2, 1), ("clike", 2, 1), ("arith", 0, ord("?"))):
        dfa, disc = T.tokenset(name), T.discarded_kinds(name)
        base = corpus.generate(name, total, seed=312)
        for pos in [0, 15, 16, 31, 32, 1023, 1024, total - 1] + [rng.randrange(total) for _ in range(3)]:
            w = base.copy()
            w[pos] = bad
            check(lg, ctx, compiled(lg, name), dfa, disc, w, mode)


def test_backtracking_at_slice_edges(env):
    # over a, a+b and ; every a that no b follows is found by failed lookahead
    # of up to the next ';': inside a slice, across one and across several
    lg, ctx = env
    dfa = T.tokenset("lookahead")
    ts = compiled(lg, "lookahead")
    rng = random.Random(6)
    for k in (1, 3, 20, 200):
        w = b"".join(b"a" * rng.randrange(1, k + 1) + rng.choice([b";", b"b;", b"b", b";;"]) for _ in range(40000 // k))
        check(lg, ctx, ts, dfa, [], w, 0)
        check(lg, ctx, ts, dfa, [], w + b"a" * k, 0, off=3)
    # an unfinished number and string at the end of the input
    dfa, disc = T.tokenset("json"), T.discarded_kinds("json")
    for tail in (b"1e", b"-", b'"abc', b"12.", b"tru"):
        for n in (31, 32, 1000, 1024):
            check(lg, ctx, compiled(lg, "json"), dfa, disc, b"[" + b"1," * ((n - len(tail)) // 2) + tail, 2)


def test_capacity_cuts_a_tile(env):
    lg, ctx = env
    dfa, disc = T.tokenset("json"), T.discarded_kinds("json")
    for n in (30_000, FUSED + 50_000):
        w = corpus.generate("json", n, seed=313)
        for cap in (0, 1, 1001, n // 10 | 1):
            check(lg, ctx, compiled(lg, "json"), dfa, disc, w, 2, cap=cap)


def test_random_automata(env):
    lg, ctx = env
    rng = random.Random(7)
    for dfa in _random_automata(606, 20, 12):
        ts = lg.lx_compile_tokenset(dfa, [])
        for n in (777, 9000):
            w = bytes(rng.choice(b"abc") for _ in range(n))
            check(lg, ctx, ts, dfa, [], w, 0, off=rng.randrange(16))


@pytest.mark.parametrize("name,mode,off,size", [("json", 2, 13, 64 << 20), ("json", 0, 0, (90 << 20) + 1001), ("arith", 0, 5, 72 << 20)])
def test_rows_found_by_the_lexing_kernel(env, name, mode, off, size):
    # csrc/rows.cu: FIND_ROUNDS; strings, spaces and digits for which a lane
    # looks 32, 128 and 512 bytes back, and an error near the end
    lg, ctx = env
    dfa, disc = T.tokenset(name), T.discarded_kinds(name)
    base = corpus.generate(name, size, seed=314)
    rng = random.Random(8)
    if name == "json":
        nl = np.flatnonzero(base == 10)
        parts, at = [], 0
        for i in range(400):
            cut = int(nl[(i + 1) * nl.size // 402]) + 1
            length = rng.choice([20, 31, 32, 33, 60, 100, 127, 128, 129, 200, 250, 300])
            parts += [base[at:cut].tobytes(), b'"' + b"z" * length + b'"\n' + b" " * rng.randrange(200)]
            at = cut
        base = np.frombuffer(b"".join(parts) + base[at:].tobytes(), np.uint8)
    check(lg, ctx, compiled(lg, name), dfa, disc, base, mode, off=off)
    bad = base.copy()
    bad[size - 5000] = ord("?")
    check(lg, ctx, compiled(lg, name), dfa, disc, bad, mode, off=off)
