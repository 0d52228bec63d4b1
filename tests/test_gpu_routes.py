"""Which kernels serve a call (lx_ctx_debug_counts), together with its tokens:
every route ends in another exact one, so that results alone do not show that
the first was taken.  And the kernels that only serve what others hand on, on
inputs that reach them: the tile kernel's configurations (LX_KERNEL_TILE) and
the 4096-byte chunks (tokens with failed lookahead on the edge of a slice)."""

import numpy as np
import pytest

import oracle
from lexinputs import corpus
from lexinputs import tokensets as T

pytestmark = pytest.mark.gpu
CH = 4096


@pytest.fixture(scope="module")
def lg(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib


def tset(lg, name):
    return lg.lx_compile_tokenset(T.tokenset(name), T.discarded_kinds(name))


def expected(name, w, mode):
    dfa = T.tokenset(name)
    k, l, con = oracle.lex(dfa, w)
    if mode:
        k, l = oracle.discard(k, l, T.discarded_kinds(name), dfa.n_kinds)
    return k, l, con


def ran(lg, ctx, before):
    """The kernels run since `before` (counts that moved)."""
    after = lg.lx_ctx_debug_counts(ctx)
    return {k: after[k] - before[k] for k in after if after[k] != before[k]}


def call(lg, ctx, name, w, mode, fn, off=0, ts=None):
    """fn(ts, d, k, l) -> (rc, tokens, consumed); checks the tokens, returns the route."""
    import torch
    w = np.frombuffer(bytes(w), np.uint8) if isinstance(w, (bytes, bytearray)) else np.ascontiguousarray(w)
    d = torch.zeros(w.size + 32, dtype=torch.uint8, device="cuda")[off:off + w.size]
    d.copy_(torch.from_numpy(w.copy()))
    k = torch.zeros(w.size + 1, dtype=torch.int16, device="cuda")
    l = torch.zeros(w.size + 1, dtype=torch.int32, device="cuda")
    before = lg.lx_ctx_debug_counts(ctx)
    rc, nt, con = fn(ts or tset(lg, name), d, k, l)[:3]
    ek, el, econ = expected(name, w, mode)
    assert rc == 0, lg.lx_strerror(rc)
    assert (nt, con) == (ek.size, econ)
    assert np.array_equal(k[:nt].cpu().numpy().view(np.uint16).astype(np.int64), ek)
    assert np.array_equal(l[:nt].cpu().numpy().view(np.uint32).astype(np.int64), el)
    return ran(lg, ctx, before)


# failed lookahead every few bytes, at all phases of a slice: "1e" before a letter
LOOKAHEAD = b"1en a; " * 900


def after_text(name, n):
    """n bytes: text, then lookahead that the entry-row kernels hand on."""
    return (corpus.generate(name, max(n - len(LOOKAHEAD), 64), seed=71).tobytes() + LOOKAHEAD)[:n]


@pytest.mark.parametrize("off", [0, 5])
@pytest.mark.parametrize("name,mode", [("json", 2), ("json", 1), ("json", 0), ("clike", 2), ("clike", 0), ("arith", 0)])
def test_lex(lg, name, mode, off):
    ctx = lg.lx_ctx_create()
    for n in (1500, 5 << 20):   # one launch, and two
        w = corpus.generate(name, n, seed=72)
        assert call(lg, ctx, name, w, mode, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, mode, k, l), off) == {"rows": 1}


def test_lex_handed_on(lg):
    # over a, a+b and ; : an a that no b follows is found by lookahead to the next ';'
    w = (b"ab;" * 5 + b"a" * 40 + b";") * 2000
    for off, route in ((0, "warps"), (3, "tiles")):
        ctx = lg.lx_ctx_create()
        for n in (5000, len(w)):
            assert call(lg, ctx, "lookahead", w[:n], 0, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 0, k, l),
                        off) == {"rows": 1, route: 1}


def test_backtracking_is_not_far(lg):
    # rows behind a token that backtracks are lost, however near the newline before it is: the old plan
    # at once, not the contexts (and then the chunks) for inputs without a newline for 8 KiB
    w = b"int a = 1en ; int b = 0;\n" * 3000
    for off, route in ((0, "warps"), (3, "tiles")):
        ctx = lg.lx_ctx_create()
        for n in (5000, len(w)):
            assert call(lg, ctx, "clike", w[:n], 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l),
                        off) == {"rows": 1, route: 1}


@pytest.mark.parametrize("length,route", [(3000, {"rows": 1}), (9000, {"rows": 1, "contexts": 1}),
                                          (17_000, {"rows": 1, "contexts": 1}), (60_000, {"rows": 1, "contexts": 1}),
                                          (80_000, {"rows": 1, "contexts": 1, "chunks": 1})])
def test_long_lines(lg, length, route):
    # C-like text synchronizes at newlines, and a comment's bytes have too many contexts for a start
    base = corpus.generate("clike", 200_000, seed=79)
    at = int(np.flatnonzero(base[:100_000] == 10)[-1]) + 1
    line = np.frombuffer(b"//" + b"c" * length + b"\n", np.uint8)
    w = np.concatenate([base[:at], line, base[at:]])
    for off in (0, 7):
        ctx = lg.lx_ctx_create()
        assert call(lg, ctx, "clike", w, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l), off) == route


def test_far_rows_that_backtrack(lg):
    # a long line and, in another tile's reach, tokens that backtrack across slices: neither the rows nor the
    # contexts serve it, the warp-tile kernel does
    base = corpus.generate("clike", 200_000, seed=80)
    at = int(np.flatnonzero(base[:100_000] == 10)[-1]) + 1
    w = np.concatenate([base[:at], np.frombuffer(b"//" + b"c" * 9000 + b"\n", np.uint8), base[at:],
                        np.frombuffer(b"\n" + b"int a = 1en ; int b = 0;\n" * 4000, np.uint8)])
    ctx = lg.lx_ctx_create()
    got = call(lg, ctx, "clike", w, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l))
    assert got in ({"rows": 1, "contexts": 1, "warps": 1}, {"rows": 1, "warps": 1})   # (which tile is met first)


def test_kernel_setting(lg):
    for kernel, route in ((lg.LX_KERNEL_TILE, "tiles"), (lg.LX_KERNEL_WARP, "warps")):
        ctx = lg.lx_ctx_create()
        assert lg.lx_ctx_set_kernel(ctx, kernel) == 0
        w = corpus.generate("json", 200_000, seed=73)
        assert call(lg, ctx, "json", w, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l)) == {route: 1}


@pytest.mark.parametrize("name", ["json", "clike"])
def test_every_tile_configuration(lg, name):
    ctx, ts = lg.lx_ctx_create(), tset(lg, name)
    assert lg.lx_ctx_set_kernel(ctx, lg.LX_KERNEL_TILE) == 0
    w = corpus.generate(name, 1 << 20, seed=74)
    for cls in (0, 1):
        for ks in (16, 24, 40, 96):
            for ctas in (0, 1):
                assert lg.lx_ctx_set_config(ctx, ts, 2, ks, ctas, cls) == 0
                assert call(lg, ctx, name, w, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l),
                            ts=ts) == {"tiles": 1}


def test_host(lg):
    import torch
    ctx, ts = lg.lx_ctx_create(), tset(lg, "json")
    for n in (1500, 25 << 20):
        w = corpus.generate("json", n, seed=75)
        k, l = torch.zeros(n, dtype=torch.int16), torch.zeros(n, dtype=torch.int32)
        before = lg.lx_ctx_debug_counts(ctx)
        rc, nt, con = lg.lx_lex_host(ctx, ts, torch.from_numpy(w.copy()), 2, k, l)
        ek, el, econ = expected("json", w, 2)
        assert rc == 0 and (nt, con) == (ek.size, econ) and np.array_equal(l[:nt].numpy().astype(np.int64), el)
        assert ran(lg, ctx, before) == {"rows": 1}


def handed_on(n, what):
    if what == "far":
        w = corpus.generate("clike", n, seed=87)
        at = int(np.flatnonzero(w[:n // 2] == 10)[-1]) + 1
        return "clike", 2, np.concatenate([w[:at], np.frombuffer(b"//" + b"c" * 9000 + b"\n", np.uint8), w[at:]])
    unit = b"ab;" * 5 + b"a" * 40 + b";"
    return "lookahead", 0, np.frombuffer(unit * (n // len(unit)), np.uint8)


@pytest.mark.parametrize("n", [20_000, 25 << 20])
@pytest.mark.parametrize("what,route", [("far", {"rows": 1, "contexts": 1}), ("backtracks", {"rows": 1, "warps": 1})])
def test_host_handed_on(lg, n, what, route):
    # one attempt on the rows, then what serves the input (refused once, the input was tried once more there)
    import torch
    name, mode, w = handed_on(n, what)
    ctx, ts = lg.lx_ctx_create(), tset(lg, name)
    k, l = torch.zeros(w.size, dtype=torch.int16), torch.zeros(w.size, dtype=torch.int32)
    before = lg.lx_ctx_debug_counts(ctx)
    rc, nt, con = lg.lx_lex_host(ctx, ts, torch.from_numpy(w.copy()), mode, k, l)
    ek, el, econ = expected(name, w, mode)
    assert rc == 0 and (nt, con) == (ek.size, econ)
    assert np.array_equal(l[:nt].numpy().astype(np.int64), el) and np.array_equal(k[:nt].numpy().astype(np.int64), ek)
    assert ran(lg, ctx, before) == route


def test_batch(lg):
    import torch
    names = ["json", "clike"]
    ctx, sets = lg.lx_ctx_create(), [tset(lg, n) for n in names]
    docs = [(i % 2, corpus.generate(names[i % 2], n, seed=76 + i)) for i, n in enumerate((100, 9000, 40000, 7, 70000))]
    d = [torch.from_numpy(w.copy()).cuda() for _, w in docs]
    k = torch.zeros(200_000, dtype=torch.int16, device="cuda")
    l = torch.zeros(200_000, dtype=torch.int32, device="cuda")
    for want in ({"rows": 1, "graphs": 1}, {"rows": 1}):
        before = lg.lx_ctx_debug_counts(ctx)
        rc, total, res = lg.lx_lex_batch(ctx, sets, [(x, s) for x, (s, _) in zip(d, docs)], 2, k, l)
        assert rc == 0 and ran(lg, ctx, before) == want
        for (s, w), (off, nt, con) in zip(docs, res):
            ek, el, econ = expected(names[s], w, 2)
            assert (nt, con) == (ek.size, econ)
            assert np.array_equal(l[off:off + nt].cpu().numpy().astype(np.int64), el)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n", [6400, 2 * CH - 1, 2 * CH, 2 * CH + 1, 3 * CH + 255, 70001, 300 * CH + 17])
def test_enumerative(lg, n, mode):
    ctx = lg.lx_ctx_create()
    for off in (0, 9):
        w = corpus.generate("clike_block", n, seed=77)
        enum = lambda ts, d, k, l: lg.lx_lex_enumerative(ctx, ts, d, mode, k, l)   # noqa: E731
        assert call(lg, ctx, "clike_block", w, mode, enum, off) == {"contexts": 1}
        # the chunks
        assert call(lg, ctx, "clike_block", after_text("clike_block", n), mode, enum, off) == {"contexts": 1, "chunks": 1}


@pytest.mark.parametrize("tiles", [1, 3, 5, 9, 14])
def test_counts_across_tiles_without_a_start(lg, tiles):
    # bytes with too many contexts for a start in whole tiles: the rounds count as the chunks' do (unaligned)
    ts, ctx = tset(lg, "clike_block"), lg.lx_ctx_create()
    base = corpus.generate("clike_block", 60_000, seed=86)
    at = int(np.flatnonzero(base[:30_000] == 10)[-1]) + 1
    w = np.concatenate([base[:at], np.frombuffer(b"//" + b"c" * (tiles * CH + 100) + b"\n", np.uint8), base[at:]])
    stats = []
    for off, route in ((0, {"contexts": 1}), (5, {"chunks": 1})):
        def spec(ts, d, k, l):
            rc, nt, con, st = lg.lx_lex_speculative(ctx, ts, None, d, 0, k, l)
            stats.append(st)
            return rc, nt, con
        assert call(lg, ctx, "clike_block", w, 0, spec, off, ts=ts) == route
    assert stats[0] == stats[1]


@pytest.mark.parametrize("with_model", [False, True])
@pytest.mark.parametrize("n", [6400, 2 * CH - 1, 2 * CH + 1, 70001, 300 * CH + 17])
def test_speculative(lg, n, with_model):
    ctx, ts = lg.lx_ctx_create(), tset(lg, "clike_block")
    model = lg.Model(lg.lx_tokenset_scan_table(ts)[2]["S"] + 1, hidden=16, seed=5) if with_model else None
    spec = lambda ts, d, k, l: lg.lx_lex_speculative(ctx, ts, model, d, 0, k, l)   # noqa: E731
    w = corpus.generate("clike_block", n, seed=78)
    assert call(lg, ctx, "clike_block", w, 0, spec, ts=ts) == {"contexts": 1}
    # the chunks: addresses that are not 16-byte aligned, and lookahead
    assert call(lg, ctx, "clike_block", w, 0, spec, off=5, ts=ts) == {"chunks": 1}
    assert call(lg, ctx, "clike_block", after_text("clike_block", n), 0, spec, ts=ts) == {"contexts": 1, "chunks": 1}


def open_ended(name, n, cut, seed):
    """A text whose last token, begun `cut` bytes before the end, has no accepting prefix."""
    base = corpus.generate(name, n, seed=seed)
    base = base[:int(np.flatnonzero(base == 10)[-1]) + 1].tobytes() if n else b""
    return base + b'"' + b"text " * (cut // 5) + b"x" * (cut % 5)


# a token that fails without an accepting prefix, begun in an earlier slice, in
# an earlier tile, many tiles before or with the input, is a lexing error at its
# start, not a reason to lex the input another way
@pytest.mark.parametrize("n,cut", [(0, 40), (0, 9000), (1000, 33), (1400, 700), (300_000, 2100), (300_000, 70_000),
                                   (5 << 20, 400), (5 << 20, 30_000)])
def test_open_token(lg, n, cut):
    ctx = lg.lx_ctx_create()
    for name in ("json", "clike"):
        if name == "clike" and cut > 8000:
            continue   # its rows are found at newlines
        w = open_ended(name, n, cut, 81)
        for off in (0, 5):
            for v in (w, w + b"\n" + corpus.generate(name, 3000, seed=82).tobytes()):   # (a raw newline ends no string)
                assert call(lg, ctx, name, v, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l), off) == {"rows": 1}


def test_batches_handed_on_keep_their_graphs(lg):
    # a batch that the rows refuse (tokens that backtrack across slices) has two graphs, each captured once:
    # alone again and again, and in turn with one that they take
    import torch
    names = ["json", "clike"]
    ctx, sets = lg.lx_ctx_create(), [tset(lg, n) for n in names]
    json = corpus.generate("json", 30_000, seed=88)
    some = np.frombuffer(b"int a = 1en ; int b = 0;\n" * 700, np.uint8)
    good = np.frombuffer(b"int a = 1e1 ; int b = 0;\n" * 700, np.uint8)
    k = torch.zeros(80_000, dtype=torch.int16, device="cuda")
    l = torch.zeros(80_000, dtype=torch.int32, device="cuda")

    def batch(second):
        d = [torch.from_numpy(w.copy()).cuda() for w in (json, second, json)]
        before = lg.lx_ctx_debug_counts(ctx)
        rc, total, res = lg.lx_lex_batch(ctx, sets, list(zip(d, (0, 1, 0))), 2, k, l)
        assert rc == 0
        for (nm, w), (off, nt, con) in zip((("json", json), ("clike", second), ("json", json)), res):
            ek, el, econ = expected(nm, w, 2)
            assert (nt, con) == (ek.size, econ)
            assert np.array_equal(l[off:off + nt].cpu().numpy().astype(np.int64), el)
        return ran(lg, ctx, before)

    first = batch(some)
    assert first["rows"] == 1 and first["warps"] == 1 and first["graphs"] <= 3   # (a buffer that grows moves both)
    batch(some)
    for _ in range(3):
        while "rows" not in batch(some):   # (refused repeatedly, not every call tries)
            pass
        while "rows" not in batch(good):
            pass
        assert batch(good) == {"rows": 1}
        assert batch(some) == {"rows": 1, "warps": 1}
        assert batch(good) == {"rows": 1}
        assert batch(some) == {"rows": 1, "warps": 1}
        assert batch(some) == {"rows": 1, "warps": 1}
        assert batch(some) == {"warps": 1}


def test_open_token_in_a_batch(lg):
    import torch
    names = ["clike", "json"]
    ctx, sets = lg.lx_ctx_create(), [tset(lg, n) for n in names]
    rng = np.random.default_rng(83)
    docs = [(i % 2, np.frombuffer(open_ended(names[i % 2], int(rng.integers(0, 60_000)), int(rng.integers(1, 3000)), 84 + i),
                                  np.uint8)) for i in range(40)]
    d = [torch.from_numpy(w.copy()).cuda() for _, w in docs]
    size = sum(w.size for _, w in docs)
    k = torch.zeros(size, dtype=torch.int16, device="cuda")
    l = torch.zeros(size, dtype=torch.int32, device="cuda")
    before = lg.lx_ctx_debug_counts(ctx)
    rc, total, res = lg.lx_lex_batch(ctx, sets, [(x, s) for x, (s, _) in zip(d, docs)], 2, k, l)
    assert rc == 0 and ran(lg, ctx, before) == {"rows": 1, "graphs": 1}
    for (s, w), (off, nt, con) in zip(docs, res):
        ek, el, econ = expected(names[s], w, 2)
        assert (nt, con) == (ek.size, econ)
        assert np.array_equal(l[off:off + nt].cpu().numpy().astype(np.int64), el)


@pytest.mark.parametrize("n,cut", [(0, 300), (5000, 400), (300_000, 150), (300_000, 9000)])
def test_open_token_from_contexts(lg, n, cut):
    ctx, ts = lg.lx_ctx_create(), tset(lg, "clike_block")
    w = open_ended("clike_block", n, cut, 85)
    assert call(lg, ctx, "clike_block", w, 2, lambda ts, d, k, l: lg.lx_lex_enumerative(ctx, ts, d, 2, k, l),
                9) == {"contexts": 1}
    stats = []
    for off, route in ((0, {"contexts": 1, "chunks": 1}), (5, {"chunks": 1})):
        def spec(ts, d, k, l):
            rc, nt, con, st = lg.lx_lex_speculative(ctx, ts, None, d, 2, k, l)
            stats.append(st)
            return rc, nt, con
        assert call(lg, ctx, "clike_block", w, 2, spec, off, ts=ts) == route
    assert stats[0] == stats[1]   # the counts of the rounds are the chunks'


@pytest.mark.parametrize("kind", ["device", "host", "batch"])
def test_repeated_refusals(lg, kind):
    # 1, 3, 7, 15, 15 calls without an attempt after the second refusal in a row and those that follow; a
    # taken input ends it
    import torch
    some = np.frombuffer(b"int a = 1en ; int b = 0;\n" * 300, np.uint8)
    good = np.frombuffer(b"int a = 1e1 ; int b = 0;\n" * 300, np.uint8)
    ctx, ts = lg.lx_ctx_create(), tset(lg, "clike")
    dev = "cpu" if kind == "host" else "cuda"
    k = torch.zeros(some.size, dtype=torch.int16, device=dev)
    l = torch.zeros(some.size, dtype=torch.int32, device=dev)
    want = {id(w): expected("clike", w, 2) for w in (some, good)}
    data = {id(w): torch.from_numpy(w.copy()).to(dev) for w in (some, good)}

    def tried(w):
        before = lg.lx_ctx_debug_counts(ctx)
        if kind == "batch":
            rc, _, ((off, nt, con),) = lg.lx_lex_batch(ctx, [ts], [(data[id(w)], 0)], 2, k, l)
        else:
            rc, nt, con = (lg.lx_lex if kind == "device" else lg.lx_lex_host)(ctx, ts, data[id(w)], 2, k, l)
        ek, el, econ = want[id(w)]
        assert rc == 0 and (nt, con) == (ek.size, econ) and np.array_equal(l[:nt].cpu().numpy().astype(np.int64), el)
        route = ran(lg, ctx, before)
        assert ("warps" in route) == (w is some or "rows" not in route)
        return route.get("rows", 0)

    calls = [tried(some) for _ in range(2 + 1 + 1 + 3 + 1 + 7 + 1 + 15 + 1 + 15 + 1)]
    assert calls == [1, 1, 0, 1, 0, 0, 0, 1] + [0] * 7 + [1] + [0] * 15 + [1] + [0] * 15 + [1]
    assert [tried(good) for _ in range(17)] == [0] * 15 + [1, 1]
    assert [tried(w) for w in (some, good, some, good, some, some, good, good)] == [1, 1, 1, 1, 1, 1, 0, 1]


@pytest.mark.parametrize("off", [0, 5])
def test_autotune_times_every_kernel(lg, off):
    # large enough that the entry-row kernels win by far; a sample that they refuse switches them off
    import torch
    w = corpus.generate("clike", 24 << 20, seed=89)
    refused = np.frombuffer(b"int a = 1en ; int b = 0;\n" * 20_000, np.uint8)
    for sample, rows in ((w, True), (refused, False)):
        ctx, ts = lg.lx_ctx_create(), tset(lg, "clike")
        d = torch.zeros(sample.size + 16, dtype=torch.uint8, device="cuda")[off:off + sample.size]
        d.copy_(torch.from_numpy(sample.copy()))
        k = torch.zeros(sample.size, dtype=torch.int16, device="cuda")
        l = torch.zeros(sample.size, dtype=torch.int32, device="cuda")
        assert lg.lx_autotune(ctx, ts, 2, d, k, l) == 0
        assert lg.lx_ctx_get_config(ctx, ts, 2)[3] > 0
        small = w[:300_000]
        route = call(lg, ctx, "clike", small, 2, lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, 2, k, l), off, ts=ts)
        assert ("rows" in route) == rows and sum(route.values()) == 1
        h = torch.from_numpy(small.copy())
        before = lg.lx_ctx_debug_counts(ctx)
        rc, nt, con = lg.lx_lex_host(ctx, ts, h, 2, torch.zeros(small.size, dtype=torch.int16),
                                     torch.zeros(small.size, dtype=torch.int32))
        assert rc == 0 and (nt, con) == (expected("clike", small, 2)[0].size, expected("clike", small, 2)[2])
        assert ("rows" in ran(lg, ctx, before)) == rows   # the same choice


@pytest.mark.parametrize("off", [0, 5])
def test_autotune_with_a_long_line(lg, off):
    # the plan that a call on such a sample takes (the entry rows, then the contexts) is what is timed: C-like
    # text on one line, which the other kernels walk with one lane
    import torch
    name, mode = "clike", 2
    lines = corpus.generate(name, 300_000, seed=92).tobytes().split(b"\n")
    w = np.frombuffer(b" ".join(x for x in lines if not any(c in x for c in (b'"', b"'", b"//"))), np.uint8)
    ctx, ts = lg.lx_ctx_create(), tset(lg, name)
    d = torch.zeros(w.size + 16, dtype=torch.uint8, device="cuda")[off:off + w.size]
    d.copy_(torch.from_numpy(w.copy()))
    k = torch.zeros(w.size, dtype=torch.int16, device="cuda")
    l = torch.zeros(w.size, dtype=torch.int32, device="cuda")
    assert lg.lx_autotune(ctx, ts, mode, d, k, l) == 0
    lex = lambda ts, d, k, l: lg.lx_lex(ctx, ts, d, mode, k, l)   # noqa: E731
    assert call(lg, ctx, name, w, mode, lex, off, ts=ts) == {"rows": 1, "contexts": 1}
