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
