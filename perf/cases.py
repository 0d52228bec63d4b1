"""The work that the performance of this library is measured on.

Every case is one call of a public entry point on inputs of the sizes and
kinds that the tests, the benchmark and the generators of this repository use:
single buffers from one small document to the 512 MiB corpus, each mode, each
kind of token set (cut at certified bytes, cut at two-byte windows, none
certified), a batch of documents, host buffers, and the gradient of the
entry-context model.  ``listed`` names the fixed ones, ``draw`` gives more of
the same ranges.

Inputs: a pool of texts of about 128 KiB made by the seeded generators, one
after the other and again from the first up to the size, the last bytes a text
of their own (each text is lexically complete, so any order of them is an
input).  The output arrays hold zeros where a call writes no token.
"""

import concurrent.futures
import functools
import math
import os

import numpy as np
import torch

import paper_2608_03473_gb300 as lg
from lexinputs import corpus, tokensets

KIB, MIB = 1 << 10, 1 << 20
PIECE = 128 * KIB       # bytes of one generated text
POOL = 192              # texts made for one input, at most
MODES = {"full": lg.LX_FULL_EXACT, "exact": lg.LX_FILTERED_EXACT, "modulo": lg.LX_FILTERED_MODULO}
# kept tokens per input byte, for the bytes that a pass has to write
KEPT = {("json", "modulo"): 0.150, ("json", "exact"): 0.150, ("json", "full"): 0.230,
        ("clike", "modulo"): 0.194, ("clike", "exact"): 0.194, ("clike", "full"): 0.303,
        ("arith", "full"): 0.505, ("clike_block", "full"): 0.274, ("clike_block", "modulo"): 0.174,
        ("clike_block_framed", "full"): 0.313}


def listed():
    return [
        # one small JSON document, as a request handler lexes it: a call's latency
        {"name": "json_1500B_modulo", "op": "lex", "corpus": "json", "mode": "modulo", "n": 1500, "offset": 0},
        # the 1 MiB arithmetic token stream of the benchmark (exact certificate, full stream)
        {"name": "arith_1M_full", "op": "lex", "corpus": "arith", "mode": "full", "n": MIB, "offset": 0},
        # the benchmark's default: one 512 MiB newline-delimited JSON buffer, whitespace discarded
        {"name": "json_512M_modulo", "op": "lex", "corpus": "json", "mode": "modulo", "n": 512 * MIB, "offset": 0},
        # exact cuts where no single byte is certified (two-byte windows), a ragged size
        {"name": "json_24M_exact", "op": "lex", "corpus": "json", "mode": "exact", "n": 24 * MIB + 7777, "offset": 0},
        # a source tree's worth of C-like text, whitespace and comments discarded
        {"name": "clike_192M_modulo", "op": "lex", "corpus": "clike", "mode": "modulo", "n": 192 * MIB, "offset": 0},
        # the same with every token kept (a formatter, a highlighter): the most output per byte
        {"name": "clike_64M_full", "op": "lex", "corpus": "clike", "mode": "full", "n": 64 * MIB + 1, "offset": 0},
        # a payload behind a header of odd length in a larger buffer: not 16-byte aligned
        {"name": "json_40M_modulo_offset5", "op": "lex", "corpus": "json", "mode": "modulo", "n": 40 * MIB, "offset": 5},
        # a token set that certifies no byte (block comments) through lx_lex
        {"name": "block_96M_modulo", "op": "lex", "corpus": "clike_block", "mode": "modulo", "n": 96 * MIB,
         "offset": 0},
        # the same kind of set through the speculative call with a trained model
        {"name": "block_160M_speculative", "op": "speculative", "corpus": "clike_block", "mode": "full",
         "n": 160 * MIB, "offset": 0, "model": True},
        # a batch of JSON and C-like documents of mixed sizes in one call
        {"name": "batch_512docs_modulo", "op": "batch", "mode": "modulo", "docs": 512, "median": 128 * KIB},
        # host buffers in, tokens back in host buffers
        {"name": "host_json_80M_modulo", "op": "host", "corpus": "json", "mode": "modulo", "n": 80 * MIB + 13},
        # loss and gradient of the entry-context model on one training batch
        {"name": "model_gradient_512", "op": "gradient", "batch": 512, "contexts": 211, "hidden": 64},
    ]


def _size(rng, lo, hi):
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    op = rng.choice(["lex"] * 9 + ["refused"] * 2 + ["speculative"] * 2 + ["batch"] * 2 + ["host", "gradient"])
    if op == "lex":
        name, mode = rng.choice([("json", "modulo"), ("json", "modulo"), ("json", "exact"), ("json", "full"),
                                 ("clike", "modulo"), ("clike", "modulo"), ("clike", "full"), ("clike", "exact"),
                                 ("arith", "full"), ("clike_block_framed", "full")])
        return {"op": "lex", "corpus": name, "mode": mode, "n": _size(rng, 1 * KIB, 256 * MIB),
                "offset": rng.choice([0, 0, 0, rng.randrange(1, 16)])}
    if op == "refused":
        return {"op": "lex", "corpus": "clike_block", "mode": rng.choice(["modulo", "full"]),
                "n": _size(rng, 256 * KIB, 128 * MIB), "offset": 0}
    if op == "speculative":
        return {"op": "speculative", "corpus": "clike_block", "mode": rng.choice(["modulo", "full"]),
                "n": _size(rng, 256 * KIB, 160 * MIB), "offset": 0, "model": rng.random() < 0.7}
    if op == "batch":
        return {"op": "batch", "mode": "modulo", "docs": _size(rng, 8, 700), "median": _size(rng, 4 * KIB, 128 * KIB)}
    if op == "host":
        return {"op": "host", "corpus": rng.choice(["json", "clike"]), "mode": "modulo",
                "n": _size(rng, 1 * KIB, 80 * MIB)}
    return {"op": "gradient", "batch": _size(rng, 64, 2048), "contexts": rng.choice([64, 128, 211]), "hidden": 64}


# ---- handles that a program keeps: the context, the compiled token sets, the trained model ----
@functools.lru_cache(maxsize=None)
def _tokenset(name):
    if name == "clike_block_framed":
        return lg.lx_compile_tokenset_framed(tokensets.tokenset("clike_block"), tokensets.discarded_kinds("clike_block"))
    return lg.lx_compile_tokenset(tokensets.tokenset(name), tokensets.discarded_kinds(name))


@functools.lru_cache(maxsize=None)
def _ctx():
    return lg.lx_ctx_create()


@functools.lru_cache(maxsize=None)
def _model():
    return lg.train_context_model(_ctx(), _tokenset("clike_block"), [_text("clike_block", 32 * MIB, 77)], hidden=64,
                                  epochs=3)


# ---- inputs ----
@functools.lru_cache(maxsize=None)
def _threads():
    return concurrent.futures.ThreadPoolExecutor(max_workers=min(16, os.cpu_count() or 1))


def _pool(name, count, rng):
    """`count` texts of the corpus, without the newlines that fill them up to PIECE bytes (but one)."""
    def one(seed):
        w = corpus.generate(name, PIECE, seed=int(seed))
        return w[:min(PIECE, int(np.flatnonzero(w != 10)[-1]) + 2)]
    return list(_threads().map(one, rng.integers(1, 1 << 62, count)))


def _text(name, n, seed, out=None):
    """n bytes of the corpus `name` as a device tensor (into `out` if given)."""
    rng = np.random.default_rng([seed, n])
    pool = _pool(name, min(n // PIECE, POOL), rng)
    d = torch.empty(n, dtype=torch.uint8, device="cuda") if out is None else out
    at = 0
    if pool:   # the whole pool as often as it fits, then its texts one by one
        whole = torch.from_numpy(np.concatenate(pool)).cuda()
        ends = np.cumsum([w.size for w in pool])
        while n - at >= whole.numel():
            d[at:at + whole.numel()].copy_(whole)
            at += whole.numel()
        fit = int(np.searchsorted(ends, n - at, side="right"))
        if fit:
            d[at:at + int(ends[fit - 1])].copy_(whole[:int(ends[fit - 1])])
            at += int(ends[fit - 1])
    if at < n:
        d[at:].copy_(torch.from_numpy(corpus.generate(name, n - at, seed=int(rng.integers(1, 1 << 62)))))
    return d


def _doc_sizes(case):
    """Document sizes (lognormal, sigma 1.66, 1 KiB to 4 MiB) and each one's corpus."""
    rng = np.random.default_rng([case["docs"], case["median"]])
    z = np.exp(math.log(case["median"]) + 1.66 * rng.standard_normal(case["docs"]))
    return np.clip(z, KIB, 4 * MIB).astype(np.int64), rng.integers(0, 2, case["docs"])


def _documents(offs, sizes, which, seed):
    """The documents' bytes: whole texts of the document's corpus, the rest a text of its own."""
    host = np.zeros(int(offs[-1]), np.uint8)
    rng = np.random.default_rng([seed, 3])
    pool = [_pool(nm, 32, rng) for nm in ("json", "clike")]
    own = rng.integers(1, 1 << 62, len(sizes))

    def fill(i):
        at, end, w = int(offs[i]), int(offs[i] + sizes[i]), int(which[i])
        j = i
        while end - at >= PIECE:
            p = pool[w][j % 32]
            host[at:at + p.size] = p
            at += p.size
            j += 1
        if at < end:
            corpus.generate(("json", "clike")[w], end - at, seed=int(own[i]), out=host[at:end])

    list(_threads().map(fill, range(len(sizes))))
    return torch.from_numpy(host)


def _capacity(n, kept):
    """Room for a quarter more tokens than such an input usually has."""
    return min(n, int(1.25 * kept * n) + 4096)


def _outputs(cap):
    return (torch.zeros(cap, dtype=torch.int16, device="cuda"), torch.zeros(cap, dtype=torch.int32, device="cuda"))


def _gradient_inputs(case, seed):
    """64-byte windows around offsets of C-like text, skewed labels, parameters."""
    rng = np.random.default_rng([seed, case["batch"]])
    b, c, h = case["batch"], case["contexts"], case["hidden"]
    text = corpus.generate("clike_block", 128 * KIB, seed=int(rng.integers(1, 1 << 62)))
    at = rng.integers(32, text.size - 32, b)
    win = text[at[:, None] + np.arange(-32, 32)].astype(np.int16)
    lab = np.minimum(rng.geometric(0.08, b) - 1, c - 1)
    lab = np.where(rng.random(b) < 0.4, c - 1, lab).astype(np.int16)
    shapes = [(257 * 8, 0.5), (32 * 40, 40 ** -0.5), (32, 0.05), (512 * h, 512 ** -0.5), (h, 0.05), (h * c, h ** -0.5),
              (c, 0.05)]
    params = np.concatenate([rng.uniform(-a, a, s) for s, a in shapes]).astype(np.float32)
    return win, lab, params


def prepare(case, seed):
    op = case["op"]
    if op == "gradient":
        win, lab, params = _gradient_inputs(case, seed)
        model = lg.Model(case["contexts"], hidden=case["hidden"])
        model.set_params(params)
        return {"op": op, "model": model, "win": torch.from_numpy(win).cuda(), "lab": torch.from_numpy(lab).cuda()}
    s = {"op": op, "ctx": _ctx(), "mode": MODES[case["mode"]]}
    if op == "batch":
        sizes, which = _doc_sizes(case)
        offs = np.concatenate([[0], np.cumsum((sizes + 15) // 16 * 16)])
        s["buf"] = _documents(offs, sizes, which, seed).cuda()
        docs = [(s["buf"][o:o + n], w) for o, n, w in zip(offs.tolist(), sizes.tolist(), which.tolist())]
        s["docs"] = lg.BatchDocs([_tokenset("json"), _tokenset("clike")], docs)
        s["kinds"], s["lens"] = _outputs(_capacity(int(offs[-1]), KEPT["clike", "modulo"]))
        return s
    s["ts"], n = _tokenset(case["corpus"]), case["n"]
    cap = _capacity(n, KEPT[case["corpus"], case["mode"]])
    if op == "host":
        s["in"] = torch.empty(n, dtype=torch.uint8).pin_memory()
        s["in"].copy_(_text(case["corpus"], n, seed))
        s["kinds"] = torch.zeros(cap, dtype=torch.int16).pin_memory()
        s["lens"] = torch.zeros(cap, dtype=torch.int32).pin_memory()
        return s
    s["in"] = torch.empty(n + 16, dtype=torch.uint8, device="cuda")[case["offset"]:case["offset"] + n]
    _text(case["corpus"], n, seed, out=s["in"])
    s["kinds"], s["lens"] = _outputs(cap)
    if op == "speculative":
        s["model"] = _model() if case["model"] else None
    return s


def run(s):
    op = s["op"]
    if op == "gradient":
        grad, loss = s["model"].gradient(s["win"], s["lab"])
        return {"gradient": grad, "loss": loss}
    if op == "lex":
        rc, nt, con = lg.lx_lex(s["ctx"], s["ts"], s["in"], s["mode"], s["kinds"], s["lens"])
    elif op == "host":
        rc, nt, con = lg.lx_lex_host(s["ctx"], s["ts"], s["in"], s["mode"], s["kinds"], s["lens"])
    elif op == "speculative":
        rc, nt, con, _ = lg.lx_lex_speculative(s["ctx"], s["ts"], s["model"], s["in"], s["mode"], s["kinds"], s["lens"])
    else:
        rc, nt, _ = lg.lx_lex_batch(s["ctx"], None, s["docs"], s["mode"], s["kinds"], s["lens"], want_results=False)
        con = np.frombuffer(s["docs"].res_arr, np.int64)   # first token, tokens and consumed bytes of every document
    if rc != lg.LX_OK:
        raise lg.LexError(rc, op)
    return {"kinds": s["kinds"], "lens": s["lens"], "tokens": nt, "consumed": con}


def work(case):
    op = case["op"]
    if op == "gradient":
        b, c, h = case["batch"], case["contexts"], case["hidden"]
        params = 257 * 8 + 32 * 40 + 32 + 512 * h + h + h * c + c
        return {"bytes": b * 130 + params * (2 + 4), "flops": 3 * 2 * b * (64 * 32 * 40 + 512 * h + h * c)}
    if op == "batch":
        sizes, which = _doc_sizes(case)
        kept = [KEPT["json", "modulo"], KEPT["clike", "modulo"]]
        return {"bytes": sum(n * (1 + 6 * kept[w]) for n, w in zip(sizes.tolist(), which.tolist())), "flops": 0}
    return {"bytes": case["n"] * (1 + 6 * KEPT[case["corpus"], case["mode"]]), "flops": 0}


def exact(case, seed):
    """The gradient and the loss in 64 bits (the products read weights rounded
    to BF16); the other cases return whole numbers."""
    if case["op"] != "gradient":
        return None
    win, lab, params = _gradient_inputs(case, seed)
    b, c, h = case["batch"], case["contexts"], case["hidden"]
    p = torch.from_numpy(params).to(torch.bfloat16).to(torch.float64).requires_grad_()
    sizes = [257 * 8, 32 * 40, 32, 512 * h, h, h * c, c]
    emb, wc, bc, w1, b1, w2, b2 = torch.split(p, sizes)
    x = torch.from_numpy(win.astype(np.int64))
    h0 = emb.view(257, 8)[x].transpose(1, 2)                                      # batch, 8, 64
    a = torch.nn.functional.conv1d(h0, wc.view(32, 5, 8).transpose(1, 2), bc, padding=2)
    m = torch.relu(a).view(b, 32, 16, 4).amax(3).transpose(1, 2).reshape(b, 512)
    z = torch.relu(m @ w1.view(512, h) + b1) @ w2.view(h, c) + b2
    loss = torch.nn.functional.cross_entropy(z, torch.from_numpy(lab.astype(np.int64)))
    grad, = torch.autograd.grad(loss, p)
    return {"gradient": grad.numpy(), "loss": float(loss.detach())}
