"""Kernels of consecutive calls overlap at their ends (dependent launches): the
same work with and without a wait for the GPU after every call gives the same
bytes, over contents that change from pass to pass, so that a read ahead of the
write before it would show.  One pass: rows appended and deposited, the block
grafted with verification on a second stream beside an append, decode of both."""
import math

import numpy as np
import pytest
import torch

import kvg_synth as syn
from kvg_testlib import dims_for, fill_canary, geometry, need_gpu, pool_u16, tables, to_dev, u16

pytestmark = pytest.mark.gpu


# one-leaf pages (two-lane hashing), 16-leaf pages (one-warp), and 1,536 of those (deposit in parts)
@pytest.mark.parametrize("geo,layers,n,fresh,passes", [("tiny", 2, 256, 3, 40), ("d128", 3, 512, 70, 20),
                                                       ("d128", 24, 2048, 200, 5)])
def test_passes_with_and_without_waits(geo, layers, n, fresh, passes):
    kvg = need_gpu()
    w = geometry(geo).with_layers(layers)
    P, scale = w.page_size, 1.0 / math.sqrt(w.head_dim)
    rows = [[x.view(torch.int16) for x in syn.kv_rows(w, n + fresh, 500 + r, "cuda")] for r in range(passes)]
    q = to_dev(syn.as_u16(syn.queries(w, layers, 1, 499)))
    pos = to_dev(syn.positions(0, n + fresh).astype(np.int32))
    parts = [[t[:, :n].contiguous() for t in kv] + [t[:, n:].contiguous() for t in kv] for kv in rows]
    torch.cuda.synchronize()

    def run(wait):
        main, side = torch.cuda.Stream(), torch.cuda.Stream()
        m, s = main.cuda_stream, side.cuda_stream
        src = kvg.Cache(dims_for(kvg, w), n // P, 1, n)
        store = kvg.Store(dims_for(kvg, w), kvg.KVG_RESIDENCY_HBM, 4 << 30)
        c = kvg.Cache(dims_for(kvg, w), n // P + -(-fresh // P), 1, n + fresh)
        fill_canary(c)
        out = torch.zeros((passes, *q.shape), dtype=q.dtype, device="cuda")
        torch.cuda.synchronize()

        def step():
            if wait:
                torch.cuda.synchronize()

        blocks = []
        for r, (k, v, fk, fv) in enumerate(parts):
            kvg.kvg_cache_release(src.h, 0, m)
            step()
            kvg.kvg_cache_append(src.h, 0, k.data_ptr(), v.data_ptr(), pos.data_ptr(), n, m)
            step()
            blocks.append(kvg.kvg_deposit(store.h, src.h, 0, 0, n, m))
            step()
            kvg.kvg_cache_release(c.h, 0, m)
            step()
            side.wait_stream(main)
            kvg.kvg_graft(store.h, blocks[-1], c.h, 0, -1, 0, kvg.KVG_GRAFT_VERIFY, s)
            step()
            kvg.kvg_cache_append(c.h, 0, fk.data_ptr(), fv.data_ptr(), pos.data_ptr() + 4 * n, fresh, m)
            step()
            main.wait_stream(side)
            kvg.kvg_decode_attention(c.h, -1, [0], q.data_ptr(), w.n_q_heads, out[r].data_ptr(), scale, m)
            step()
        torch.cuda.synchronize()
        kvg.kvg_sync(c.h)  # raises on any mismatch of a verified graft
        return ([u16(out), pool_u16(c, w), *tables(c)],
                [kvg.kvg_store_export(store.h, b) for b in blocks])

    plain, overlapped = run(True), run(False)
    for a, b in zip(plain[0], overlapped[0]):
        assert np.array_equal(a, b)
    assert plain[1] == overlapped[1]
    assert len({o.tobytes() for o in plain[0][0]}) == passes
