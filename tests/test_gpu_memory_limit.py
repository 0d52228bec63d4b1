"""Calls when little device memory is left: the entry contexts' maps take 0.2
bytes per input byte, the 4096-byte chunks 0.06, so what the chunks can serve
is served."""

import numpy as np
import pytest

from lexinputs import corpus
from lexinputs import tokensets as T

pytestmark = pytest.mark.gpu
MIB = 1 << 20


def test_enumerative_without_room_for_the_maps(lexlib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lg = lexlib
    ts = lg.lx_compile_tokenset(T.tokenset("clike_block"), T.discarded_kinds("clike_block"))
    text = corpus.generate("clike_block", 8 * MIB, seed=90)
    text = text[:int(np.flatnonzero(text == 10)[-1]) + 1]
    d = torch.from_numpy(np.tile(text, 64)).cuda()
    k = torch.zeros(1000, dtype=torch.int16, device="cuda")
    l = torch.zeros(1000, dtype=torch.int32, device="cuda")

    def lex(ctx, n):
        before = lg.lx_ctx_debug_counts(ctx)
        rc, nt, con = lg.lx_lex_enumerative(ctx, ts, d, 2, k, l, n=n)
        after = lg.lx_ctx_debug_counts(ctx)
        return rc, nt, con, l.cpu().numpy().tolist(), {x: after[x] - before[x] for x in after if after[x] != before[x]}

    plenty = lg.lx_ctx_create()
    want = lex(plenty, d.numel())
    assert want[0] == lg.LX_E_CAPACITY and want[2] == d.numel() and want[4] == {"contexts": 1}
    del plenty
    ctx = lg.lx_ctx_create()
    # both routes once on little input (their kernels are loaded then)
    d[3000:9300].copy_(torch.from_numpy(np.frombuffer(b"1en a; " * 900, np.uint8).copy()))
    assert lex(ctx, 20_000)[4] == {"contexts": 1, "chunks": 1}
    d[:10_000].copy_(torch.from_numpy(text[:10_000].copy()))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = 75 * MIB   # the maps: 103 MiB, the chunks: 31
    hog = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        got = lex(ctx, d.numel())
        assert got[:4] == want[:4] and got[4] == {"chunks": 1}
        d[:20_000].copy_(torch.from_numpy(corpus.generate("clike_block", 20_000, seed=91)))
        assert lex(ctx, 20_000)[4] == {"contexts": 1}   # and nothing is left behind
    finally:
        del hog
        torch.cuda.empty_cache()
