"""lx_lex_enumerative from enumerated entry contexts (csrc/ctxmap.cu) against
the oracle: sizes at the edges of slices, tiles and of the windows in which
starts are searched, every input alignment, starts with more candidates than
one walk takes, backtracking at every phase of a slice, inputs it hands to the
chunks of csrc/enumerate.cu, and the speculative call's counts on inputs
whose rounds are known."""

import random

import numpy as np
import pytest

import oracle
from lexinputs import corpus
from lexinputs import tokensets as T
from lexinputs.automaton import Token, compile_tokens

from test_oracle_bruteforce import _random_automata

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib, lexlib.lx_ctx_create()


def check(lg, ctx, ts, dfa, disc, w, mode, off=0):
    import torch
    w = np.frombuffer(bytes(w), np.uint8) if isinstance(w, (bytes, bytearray)) else np.ascontiguousarray(w)
    n = int(w.size)
    d = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")[off:off + n]
    d.copy_(torch.from_numpy(w.copy()))
    k = torch.zeros(n + 1, dtype=torch.int16, device="cuda")
    l = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rc, nt, con = lg.lx_lex_enumerative(ctx, ts, d, mode, k, l, n=n)
    ek, el, econ = oracle.lex(dfa, w)
    if mode:
        ek, el = oracle.discard(ek, el, disc, dfa.n_kinds)
    assert rc == 0, lg.lx_strerror(rc)
    assert (nt, con) == (ek.size, econ)
    assert np.array_equal(k[:nt].cpu().numpy().view(np.uint16).astype(np.int64), ek)
    assert np.array_equal(l[:nt].cpu().numpy().view(np.uint32).astype(np.int64), el)


@pytest.mark.parametrize("n", [1, 16, 63, 64, 65, 127, 128, 129, 4095, 4096, 4097, 4096 + 255, 3 * 4096 + 128, 70001])
def test_sizes_and_alignment(env, n):
    lg, ctx = env
    dfa, disc = T.tokenset("clike_block"), T.discarded_kinds("clike_block")
    ts = lg.lx_compile_tokenset(dfa, disc)
    w = corpus.generate("clike_block", 80_000, seed=401)[:n]
    for off in (0, 1, 9):
        for mode in (0, 2):
            check(lg, ctx, ts, dfa, disc, w, mode, off=off)


def test_many_candidates(env):
    # over keyword-like tokens every letter has many contexts: starts with seven
    # and eight candidates, and stretches where no byte has few enough
    lg, ctx = env
    rng = random.Random(8)
    words = ["abcabc", "bcaabc", "cababc", "abcbca", "cbacba", "aabbcc", "ccbbaa"]
    toks = [Token("kw_" + w, w, 0) for w in words] + [Token("id", "[a-c]+", 1), Token("str", '"[a-c ]*"', 1),
                                                      Token("ws", "[ ]+", 1)]
    dfa = compile_tokens(toks)
    ts = lg.lx_compile_tokenset(dfa, [])
    w = b"".join(rng.choice([b"abc", b"abcabc", b"cab", b" ", b'"ab c"', b"ccbbaa ", b"b"]) for _ in range(20000))
    for mode in (0, 1):
        check(lg, ctx, ts, dfa, [], w, mode)
    check(lg, ctx, ts, dfa, [], bytes(rng.choice(b"abc") for _ in range(60000)), 0)


def test_backtracking_phases(env):
    # "1e" and ".." end in failed lookahead of one byte, at every offset of a slice
    lg, ctx = env
    dfa, disc = T.tokenset("clike_block"), T.discarded_kinds("clike_block")
    ts = lg.lx_compile_tokenset(dfa, disc)
    for shift in range(0, 130, 3):
        line = b"x = 1en + a..b; y = 0xg;\n"
        w = b" " * shift + line * 400
        check(lg, ctx, ts, dfa, disc, w, 2 if shift % 2 else 0)
    # a comment, a string and a character that never close
    base = corpus.generate("clike_block", 30_000, seed=402).tobytes()
    for tail in (b"\n/* open", b'\nx = "open', b"\nc = 'open\n x"):
        for n in (5000, 29_000):
            check(lg, ctx, ts, dfa, disc, base[:n] + tail, 2)


def test_random_automata(env):
    lg, ctx = env
    rng = random.Random(9)
    for dfa in _random_automata(707, 20, 12):
        ts = lg.lx_compile_tokenset(dfa, [])
        for n in (500, 9000):
            check(lg, ctx, ts, dfa, [], bytes(rng.choice(b"abc") for _ in range(n)), 0, off=rng.randrange(16))


def test_speculative_counts(env):
    # without a model every chunk starts at BOUNDARY: chunk starts inside one
    # long comment are wrong, and the fix-up moves one chunk a round
    import torch
    lg, ctx = env
    dfa, disc = T.tokenset("clike_block"), T.discarded_kinds("clike_block")
    ts = lg.lx_compile_tokenset(dfa, disc)
    code = (b"int a = b;\n" * 2000)[:5 * 4096 + 900]
    body = b"text in a comment\n" * 2000
    for chunks in (1, 3):
        w = np.frombuffer(code[:-1] + b"\n/*" + body[:chunks * 4096] + b"*/\n" + code, np.uint8)
        d = torch.from_numpy(w.copy()).cuda()
        k = torch.zeros(w.size, dtype=torch.int16, device="cuda")
        l = torch.zeros(w.size, dtype=torch.int32, device="cuda")
        rc, nt, con, st = lg.lx_lex_speculative(ctx, ts, None, d, 0, k, l)
        ek, el, econ = oracle.lex(dfa, w)
        assert rc == 0 and (nt, con) == (ek.size, econ)
        assert np.array_equal(l[:nt].cpu().numpy().view(np.uint32).astype(np.int64), el)
        inside = [j for j in range(1, -(-w.size // 4096)) if len(code) + 2 <= j * 4096 < len(code) + chunks * 4096]
        assert st["chunks"] == -(-w.size // 4096) and not st["judged"]
        assert st["rescanned"] >= len(inside) and st["rounds"] >= 1 + len(inside)


@pytest.mark.parametrize("tiles", [1023, 1024, 1025, 2049])
def test_tile_maps_across_blocks(env, tiles):
    # csrc/ctxmap.cu: cm_fold, cm_top compose 1024 tiles a block
    lg, ctx = env
    dfa, disc = T.tokenset("clike_block"), T.discarded_kinds("clike_block")
    ts = lg.lx_compile_tokenset(dfa, disc)
    w = corpus.generate("clike_block", tiles * 4096 - 9, seed=403).copy()
    w[500:502] = np.frombuffer(b"/*", np.uint8)   # at the latest the next "*/" closes it
    check(lg, ctx, ts, dfa, disc, w, 2)
    w = np.frombuffer(b"/* " + b"in a comment\n" * (tiles * 4096 // 13) + b"*/ int a;\n", np.uint8)
    check(lg, ctx, ts, dfa, disc, w, 0)
