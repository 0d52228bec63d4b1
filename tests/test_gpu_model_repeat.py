"""The dense layers' gradients (W1, b1, W2, b2) and the loss are the same each
time they are computed: their sums over the batch have an order of their own,
whatever the order in which the slices of the batch finish.  (The embedding's
and the filters' gradients are summed as they come, and the loss as well past
256 hidden units.)"""

import numpy as np
import pytest

from lexinputs import corpus
from oracle import model as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hidden,contexts", [(64, 64, 211), (65, 64, 211), (512, 64, 211), (513, 100, 65),
                                                   (1025, 64, 211), (2048, 64, 128), (4100, 256, 300), (512, 257, 40)])
def test_dense_gradients_repeat(lexlib, batch, hidden, contexts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(batch)
    m = lexlib.Model(contexts, hidden=hidden, seed=17)
    w = corpus.generate("clike_block", 1 << 17, seed=504)
    win = OM.windows(w, np.sort(rng.integers(0, w.size, size=batch)))
    dw = torch.from_numpy(win.astype(np.int16)).cuda()
    dy = torch.from_numpy(rng.integers(0, contexts, size=batch).astype(np.int16)).cuda()
    dense = sum(OM.sizes(hidden, contexts)[:3])
    first, loss = m.gradient(dw, dy)
    first = first[dense:].copy()
    assert np.all(np.isfinite(first)) and np.any(first != 0)
    for _ in range(30):
        g, l = m.gradient(dw, dy)
        assert np.array_equal(g[dense:], first)
        assert hidden > 256 or l == loss
    if hidden <= 256:   # a mean in 64 bits of losses that are each within a few units in the last place
        z, _ = OM.forward(OM.to_bf16(m.get_params().astype(np.float64)), win, hidden, contexts)
        zmax = z.max(1, keepdims=True)
        want = np.mean(np.log(np.exp(z - zmax).sum(1)) + zmax[:, 0] - z[np.arange(batch), dy.cpu().numpy()])
        assert abs(loss - want) <= 4 * np.spacing(np.float32(want))
