"""Deposits whose digests are computed in parts (chunks of pages, their page
digests and the block digest's chain side by side) give the oracle's bytes at
the sizes where the split changes: one chunk, just past one, a short last
chunk, several growing chunks; with odd and even counts of position tags, so
that a chunk's end falls inside a 64-byte block of the chain; into an HBM and
a pinned-host store."""
import numpy as np
import pytest
import torch

import kvg_synth as syn
from kvg_testlib import append, dims_for, need_gpu, oracle_dims

pytestmark = pytest.mark.gpu


# one-leaf pages (4 KiB): a wave is 152 x 128 = 19,456 of them, in 2 x 16 planes 608 pages
@pytest.mark.parametrize("tokens", [600 * 16, 608 * 16 + 760 * 16 // 4, 800 * 16 + 5, 1000 * 16 + 2, 1900 * 16 + 1])
@pytest.mark.parametrize("residency", [0, 1])
def test_deposit_parts_match_oracle(oracle, tokens, residency):
    kvg = need_gpu()
    w = syn.Workload("parts", 16, 2, 2, 64, 16, 10000.0, 0x68)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, tokens, 69))
    pos = syn.positions(3, tokens)
    c = kvg.Cache(dims_for(kvg, w), -(-tokens // 16), 1, tokens)
    append(kvg, c, 0, k, v, pos)
    store = kvg.Store(dims_for(kvg, w), residency, 4 << 30)
    first = kvg.kvg_deposit(store.h, c.h, 0, 0, tokens)
    again = kvg.kvg_deposit(store.h, c.h, 0, 0, tokens)  # right behind: shares scratch and streams
    want = oracle.block_from_kv(oracle_dims(oracle, w), k, v, pos).serialize()
    assert kvg.kvg_store_export(store.h, first) == want
    assert kvg.kvg_store_export(store.h, again) == want
    rep = kvg.kvg_graft_report()
    kvg.kvg_cache_release(c.h, 0)
    kvg.kvg_graft(store.h, again, c.h, 0, -1, 0, kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC, report=rep)
    assert rep.n_mismatch == 0
    torch.cuda.synchronize()
    assert np.frombuffer(want[96:128], np.uint8).any()
