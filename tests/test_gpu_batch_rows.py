"""lx_lex_batch from entry rows (csrc/rows.cu) against the oracle, document by
document: lengths at the edges of slices and tiles, one-byte and empty
documents, documents of one token longer than many tiles, lexing errors in the
first, a middle and the last document, both kinds of token set interleaved,
one set alone, and a batch whose rows do not fit (handed to the other form)."""

import random

import numpy as np
import pytest

import oracle
from lexinputs import corpus
from lexinputs import tokensets as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lg = lexlib
    ts = {n: lg.lx_compile_tokenset(T.tokenset(n), T.discarded_kinds(n)) for n in ("json", "clike", "lookahead")}
    return lg, lg.lx_ctx_create(), ts


def check(lg, ctx, ts, names, docs, mode=2):
    import torch
    offs, at = [], 0
    for _, w in docs:
        offs.append(at)
        at += (len(w) + 15) // 16 * 16
    host = np.zeros(at + 16, np.uint8)
    for o, (_, w) in zip(offs, docs):
        host[o:o + len(w)] = np.frombuffer(bytes(w), np.uint8)
    d = torch.from_numpy(host).cuda()
    k = torch.zeros(at + 16, dtype=torch.int16, device="cuda")
    l = torch.zeros(at + 16, dtype=torch.int32, device="cuda")
    items = [(d[o:o + len(w)], names.index(nm)) for o, (nm, w) in zip(offs, docs)]
    for _ in range(2):   # the captured graph, then its replay
        rc, total, res = lg.lx_lex_batch(ctx, [ts[n] for n in names], items, mode, k, l)
        assert rc == 0, lg.lx_strerror(rc)
        kk, ll = k.cpu().numpy().view(np.uint16), l.cpu().numpy().view(np.uint32)
        end = 0
        for (nm, w), (off, nt, con) in zip(docs, res):
            if not len(w):
                assert (off, nt, con) == (0, 0, 0)
                continue
            ek, el, econ = oracle.lex(T.tokenset(nm), bytes(w))
            if mode:
                ek, el = oracle.discard(ek, el, T.discarded_kinds(nm), T.tokenset(nm).n_kinds)
            assert (nt, con) == (ek.size, econ), (nm, len(w))
            assert mode == 0 or off >= end   # (the other form may order the documents by set)
            end = off + nt
            assert np.array_equal(kk[off:end].astype(np.int64), ek) and np.array_equal(ll[off:end].astype(np.int64), el)
        assert mode == 0 or total >= end, (total, end)


def text(nm, n, seed):
    return corpus.generate(nm, n, seed=seed).tobytes()


def test_lengths(env):
    lg, ctx, ts = env
    lengths = [1, 0, 2, 15, 16, 17, 127, 128, 129, 191, 192, 1023, 1024, 1025, 0, 4096, 6143, 6144, 6145, 7168, 8192, 20001]
    docs = [(("json", "clike")[i % 2], text(("json", "clike")[i % 2], n, 600 + i)) for i, n in enumerate(lengths)]
    check(lg, ctx, ts, ["json", "clike"], docs)
    check(lg, ctx, ts, ["json", "clike"], docs, mode=0)
    check(lg, ctx, ts, ["clike"], [(nm, w) for nm, w in docs if nm == "clike"])
    check(lg, ctx, ts, ["json", "clike"], [("json", text("json", 3, 1))])


def test_long_tokens_and_errors(env):
    lg, ctx, ts = env
    rng = random.Random(3)
    big = b'["' + b"z" * 40000 + b'",\n' + b" " * 20000 + b"1]\n"
    docs = [("json", text("json", 5000, 1)), ("json", big), ("clike", b"// " + b"c" * 30000 + b"\nint a;\n"),
            ("clike", text("clike", 9000, 2)), ("json", big + text("json", 9000, 3))]
    check(lg, ctx, ts, ["json", "clike"], docs)
    for bad in ([0], [2, 3], [4], [0, 4]):
        d2 = []
        for i, (nm, w) in enumerate(docs):
            w = bytearray(w)
            if i in bad:
                w[rng.randrange(len(w))] = 1
            d2.append((nm, bytes(w)))
        check(lg, ctx, ts, ["json", "clike"], d2)


def test_many_small_and_handed_over(env):
    lg, ctx, ts = env
    rng = random.Random(4)
    docs = []
    for i in range(700):
        nm = rng.choice(["json", "clike"])
        docs.append((nm, text(nm, rng.choice([5, 40, 300, 1500, 9000]), i)))
    check(lg, ctx, ts, ["clike", "json"], docs)
    # no synchronizing byte for thousands of bytes, and failed lookahead across slices
    check(lg, ctx, ts, ["json", "lookahead"], docs[:0] + [("lookahead", b"a" * 9000 + b";" + b"a" * 700 + b"b;"),
                                                           ("json", text("json", 3000, 5))], mode=0)
