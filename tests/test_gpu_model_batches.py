"""The context model's gradient and loss against the FP64 reference at the
BF16-rounded weights: batches at the edges of the windows one CTA takes and of
the batch slices of the weight gradients, layer sizes at the edges of their
tiles, up to and past the sizes of the fused kernel, and windows of one
repeated byte and of padding.  FP32 sums of at most a few thousand terms:
tolerances as in test_gpu_speculative.py."""

import numpy as np
import pytest

from lexinputs import corpus
from oracle import model as OM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lg(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib


@pytest.mark.parametrize("batch,hidden,contexts", [
    (1, 64, 211), (3, 64, 211), (4, 64, 211), (5, 16, 2), (63, 64, 64), (64, 32, 65), (65, 64, 63), (130, 1, 33),
    (257, 100, 300), (8, 256, 1024), (8, 257, 40), (8, 40, 1025)])
def test_gradient_sizes(lg, batch, hidden, contexts):
    import torch
    rng = np.random.default_rng(batch * 7 + hidden)
    m = lg.Model(contexts, hidden=hidden, seed=11)
    w = corpus.generate("clike_block", 1 << 16, seed=501)
    pos = np.sort(rng.integers(0, w.size, size=batch))
    win = OM.windows(w, pos)
    win[0] = 256                       # padding alone
    if batch > 2:
        win[1] = 32                    # one byte value: every position adds to the same embedding row
    y = rng.integers(0, contexts, size=batch)
    p = OM.to_bf16(m.get_params().astype(np.float64))
    dw = torch.from_numpy(win.astype(np.int16)).cuda()
    dy = torch.from_numpy(y.astype(np.uint16).view(np.int16)).cuda()
    rl, rg = OM.loss_and_grad(p, win, y, hidden, contexts)
    for _ in range(2):                 # and again on used buffers
        g, loss = m.gradient(dw, dy)
        assert abs(loss - rl) < 1e-4 * (1 + abs(rl))
        blocks = np.cumsum([0] + OM.sizes(hidden, contexts))
        for lo, hi in zip(blocks[:-1], blocks[1:]):
            assert np.max(np.abs(g[lo:hi] - rg[lo:hi])) < 1e-5 + 1e-3 * np.max(np.abs(rg[lo:hi])), (lo, hi)
    z = m.forward(dw).cpu().numpy()
    rz, _ = OM.forward(p, win, hidden, contexts)
    assert np.max(np.abs(z - rz)) < 1e-4 * (1 + np.max(np.abs(rz)))


def test_step_equals_its_gradient(lg):
    # the first AdamW step moves every weight by lr against its gradient's sign
    import torch
    rng = np.random.default_rng(5)
    m = lg.Model(40, hidden=32, seed=12)
    w = corpus.generate("clike_block", 1 << 14, seed=502)
    win = OM.windows(w, np.sort(rng.integers(0, w.size, size=48)))
    y = rng.integers(0, 40, size=48)
    dw = torch.from_numpy(win.astype(np.int16)).cuda()
    dy = torch.from_numpy(y.astype(np.int16)).cuda()
    p0 = m.get_params()
    g, loss = m.gradient(dw, dy)
    assert abs(m.train_step(dw, dy, 1e-3) - loss) < 1e-5 * (1 + abs(loss))
    big = np.abs(g) > 1e-4
    step = (m.get_params() - p0)[big]
    assert big.sum() > 1000 and np.all(np.sign(step) == -np.sign(g[big]))
    assert np.max(np.abs(np.abs(step) - 1e-3)) < 1e-5


@pytest.mark.parametrize("chunks,hidden", [(2, 64), (63, 33), (64, 64), (65, 64), (1001, 100), (24579, 64)])
def test_predictions_of_a_speculative_call(lg, chunks, hidden):
    # a model whose argmax (by lx_model_forward, other kernels) is the true
    # context at the chunk starts of a text of three chunks, repeated: nothing
    # is scanned again
    import torch
    from lexinputs import tokensets as T
    ts = lg.lx_compile_tokenset(T.tokenset("clike_block"), T.discarded_kinds("clike_block"))
    _, blob, t = lg.lx_tokenset_scan_table(ts)
    cbeg = blob[t["cbeg_off"]:t["cbeg_off"] + 514].view(np.uint16).astype(np.int64)
    cands = blob[t["cand_off"]:t["cand_off"] + 2 * int(cbeg[256])].view(np.uint16).astype(np.int64)
    text = corpus.generate("clike_block", 60_000, seed=31)
    text = text[:int(np.flatnonzero(text[:3 * 4096 - 40] == 10)[-1]) + 1]
    text = np.concatenate([text, np.full(3 * 4096 - text.size, ord(" "), np.uint8)])
    w = np.resize(text, chunks * 4096 - 100)
    d = torch.from_numpy(w.copy()).cuda()
    ctx = lg.lx_ctx_create()
    rc, starts, labels = lg.lx_chunk_contexts(ctx, ts, d)
    assert rc == 0
    starts, labels = starts.cpu().numpy(), labels.cpu().numpy().view(np.uint16).astype(np.int64)
    assert starts.size == chunks and (starts >= 0).all()
    some = np.arange(1, min(chunks, 7))
    for seed in range(1, 2000):
        m = lg.Model(t["S"] + 1, hidden=hidden, seed=seed)
        z = m.forward(m.windows(d, torch.from_numpy(starts[some].astype(np.int64)).cuda())).cpu().numpy()
        for j, v in zip(some, z):
            b = int(w[starts[j] - 1])
            c = np.append(np.sort(cands[cbeg[b]:cbeg[b + 1]]), t["S"])
            order = np.argsort(-v[c])
            best = c[order[0]]
            if (lg.CTX_BOUNDARY if best == t["S"] else best) != labels[j] or (
                    order.size > 1 and v[c[order[0]]] - v[c[order[1]]] < 1e-4):
                break
        else:
            break
    else:
        pytest.fail("no seed predicts the text")
    k = torch.zeros(w.size, dtype=torch.int16, device="cuda")
    l = torch.zeros(w.size, dtype=torch.int32, device="cuda")
    rc, nt, con, st = lg.lx_lex_speculative(ctx, ts, m, d, 0, k, l)
    assert rc == 0 and con == w.size
    assert (st["chunks"], st["rescanned"], st["rounds"]) == (chunks, 0, 1)
