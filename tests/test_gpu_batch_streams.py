"""Batches of grafts into different sequences of one cache on two streams: the
later batch's job table must not replace the earlier one's while its copy runs.
Pages, tables and tags equal the same batches one after another on one stream."""
import numpy as np
import pytest
import torch

import kvg_synth as syn
from kvg_testlib import append, dims_for, fill_canary, geometry, need_gpu, pool_u16, tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geo,layers,lens", [("tiny", 4, [900, 37, 400, 16]), ("d128", 8, [1500, 64, 777, 65])])
def test_two_streams_keep_their_job_tables(geo, layers, lens):
    kvg = need_gpu()
    w = geometry(geo).with_layers(layers)
    P = w.page_size
    src = kvg.Cache(dims_for(kvg, w), max(-(-n // P) for n in lens), 1, max(lens))
    store = kvg.Store(dims_for(kvg, w), kvg.KVG_RESIDENCY_HBM, 2 << 30)
    bids = []
    for i, n in enumerate(lens):
        k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 410 + i))
        append(kvg, src, 0, k, v, syn.positions(0, n))
        bids.append(kvg.kvg_deposit(store.h, src.h, 0, 0, n))
        kvg.kvg_cache_release(src.h, 0)
    torch.cuda.synchronize()
    per_seq = sum(-(-n // P) for n in lens)
    caches = []
    for _ in range(2):
        c = kvg.Cache(dims_for(kvg, w), 4 * per_seq, 4, per_seq * P)
        fill_canary(c)
        caches.append(c)
    n = len(lens)
    # (own positions, re-based) x (long, short): a short batch follows a long one
    batches = [(0, bids, [0] * n), (1, bids[1:2], [0]), (2, bids[::-1], [7, 0, 1000, 7]), (3, bids[3:], [19])]
    streams = [torch.cuda.Stream() for _ in range(2)]
    for rep in range(8):
        for j, c in enumerate(caches):
            for i, (seq, blocks, deltas) in enumerate(batches):
                st = streams[i % 2 if j else 0].cuda_stream
                kvg.kvg_graft_batch(store.h, blocks, c.h, [seq] * len(blocks), 0, st, deltas=deltas)
            torch.cuda.synchronize()
        assert np.array_equal(pool_u16(caches[0], w), pool_u16(caches[1], w)), rep
        for a, b in zip(tables(caches[0]), tables(caches[1])):
            assert np.array_equal(a, b), rep
        for c in caches:
            for seq in range(4):
                kvg.kvg_cache_release(c.h, seq)
            torch.cuda.synchronize()
