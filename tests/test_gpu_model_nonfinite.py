"""The context model's gradient with infinities and NaN among the parameters
(a run that has diverged)."""

import numpy as np
import pytest

from lexinputs import corpus
from oracle import model as OM

pytestmark = pytest.mark.gpu
C, H = 211, 64


@pytest.fixture(scope="module")
def lg(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lexlib


def batch(n, seed):
    import torch
    rng = np.random.default_rng(seed)
    w = corpus.generate("clike_block", 1 << 14, seed=503)
    win = OM.windows(w, np.sort(rng.integers(32, w.size - 32, size=n)))
    y = rng.integers(0, C, size=n)
    return win, torch.from_numpy(win.astype(np.int16)).cuda(), torch.from_numpy(y.astype(np.int16)).cuda()


def parameters(block, at, value, seed=13):
    rng = np.random.default_rng(seed)
    p = [rng.uniform(-0.3, 0.3, n).astype(np.float32) for n in OM.sizes(H, C)]
    p[block][at] = value
    return p


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7])
def test_rows_of_other_bytes_take_nothing(lg, n):
    # an infinite filter weight makes NaN of the zeros where no window stands
    # (four windows a CTA): no embedding row but the windows' own may see it
    win, dw, dy = batch(n, n)
    m = lg.Model(C, hidden=H)
    m.set_params(np.concatenate(parameters(1, 77, np.inf)))
    g, _ = m.gradient(dw, dy)
    rows = g[:OM.ROWS * OM.D].reshape(OM.ROWS, OM.D)
    others = np.setdiff1d(np.arange(OM.ROWS), win)
    assert others.size > 100 and np.all(rows[others] == 0)


WIDE = 257   # past the sizes of the one-kernel form: the layers' kernels one by one


def widened(p):
    """The same function with WIDE hidden units: the rest of weight zero."""
    emb, wc, bc, w1, b1, w2, b2 = p
    return np.concatenate([emb, wc, bc, np.pad(w1.reshape(-1, H), ((0, 0), (0, WIDE - H))).ravel(),
                           np.pad(b1, (0, WIDE - H)), np.pad(w2.reshape(H, C), ((0, WIDE - H), (0, 0))).ravel(), b2])


def narrowed(g):
    emb, wc, bc, w1, b1, w2, b2 = np.split(g, np.cumsum(OM.sizes(WIDE, C))[:-1])
    return [emb, wc, bc, w1.reshape(-1, WIDE)[:, :H].ravel(), b1[:H], w2.reshape(WIDE, C)[:H].ravel(), b2]


def check_against_the_layers(lg, p, n):
    """Gradient and loss equal those of the general kernels: NaN and infinities
    in the same places, finite values within the tolerance of the FP32 sums."""
    win, dw, dy = batch(n, 100 + n)
    m, wide = lg.Model(C, hidden=H), lg.Model(C, hidden=WIDE)
    m.set_params(np.concatenate(p))
    wide.set_params(widened(p))
    g, loss = m.gradient(dw, dy)
    rg, rl = wide.gradient(dw, dy)
    assert np.isnan(loss) == np.isnan(rl) and (np.isnan(rl) or abs(loss - rl) < 1e-4 * (1 + abs(rl)))
    for i, (a, b) in enumerate(zip(np.split(g, np.cumsum(OM.sizes(H, C))[:-1]), narrowed(rg))):
        assert np.array_equal(np.isnan(a), np.isnan(b)), i
        assert np.array_equal(np.isinf(a), np.isinf(b)), i
        ok = np.isfinite(b)
        if ok.any():
            assert np.max(np.abs(a[ok] - b[ok])) < 1e-5 + 1e-3 * np.max(np.abs(b[ok])), i
    return loss


@pytest.mark.parametrize("n", [1, 4, 6, 65])
@pytest.mark.parametrize("block,at,value", [(3, 5 * H + 3, np.nan), (4, 3, np.nan), (5, 3 * C + 2, np.nan), (6, 2, np.nan),
                                            (4, 3, np.inf), (4, 3, -np.inf), (5, 3 * C + 2, np.inf)])
def test_dense_layers_keep_nan(lg, block, at, value, n):
    loss = check_against_the_layers(lg, parameters(block, at, value), n)
    if np.isnan(value):
        assert np.isnan(loss)


@pytest.mark.parametrize("n", [1, 4, 6, 65])
@pytest.mark.parametrize("block,at,value", [(0, 32 * 8 + 1, np.nan), (0, 101 * 8, np.inf), (0, 101 * 8 + 5, -np.inf),
                                            (1, 77, np.nan), (1, 77, np.inf), (1, 78, -np.inf), (2, 3, np.nan),
                                            (2, 3, np.inf), (2, 3, -np.inf)])
def test_inactive_positions_add_nothing(lg, block, at, value, n):
    # embedding, filters, their bias: a convolution output of NaN is no maximum
    loss = check_against_the_layers(lg, parameters(block, at, value), n)
    if np.isnan(value):
        assert np.isfinite(loss)
