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


# one-leaf pages (4 KiB): with 152 SMs a chunk starts at (152 - 8) x 128 = 18,432
# of them, 576 pages in each of the 2 x 16 planes, and a block is hashed in chunks
# from 720 on
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


# kv heads, head_dim, page size, layers, tokens
@pytest.mark.parametrize("hkv,d,page,layers,tokens,parts", [
    (8, 256, 128, 20, 4 * 128 + 9, True),    # 128 leaves a page
    (8, 256, 256, 26, 256 + 3, True),        # 256, the most that is hashed in parts
    (8, 256, 512, 16, 512 + 1, False),       # 512: one after the other
    (3, 128, 17, 40, 73 * 17 - 3, True),     # three leaves and one of 768 bytes
    (8, 256, 64, 185, 1, True),              # few position tags: the chain's first parts are
    (8, 256, 64, 185, 7, True),              # empty, and a later one starts it in the middle
    (8, 256, 64, 185, 15, True),             # of a block of tags and digests
    (8, 256, 64, 185, 16, True),
    (8, 256, 64, 185, 20, True),
])
def test_deposit_of_large_pages_and_few_tags(oracle, hkv, d, page, layers, tokens, parts):
    kvg = need_gpu()
    w = syn.Workload("large", layers, hkv, hkv, d, page, 10000.0, 0x69)
    leaves = -(-w.page_bytes // 4096)
    chunk = max(1, (torch.cuda.get_device_properties(0).multi_processor_count - 8) * 128 // leaves)
    pages = -(-tokens // page)
    assert (2 * layers * pages > chunk + chunk // 4 and leaves <= 256) == parts
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, tokens, 70))
    pos = syn.positions(3, tokens)
    c = kvg.Cache(dims_for(kvg, w), pages, 1, pages * page)
    append(kvg, c, 0, k, v, pos)
    store = kvg.Store(dims_for(kvg, w), kvg.KVG_RESIDENCY_HBM, 1 << 30)
    bid = kvg.kvg_deposit(store.h, c.h, 0, 0, tokens)
    want = oracle.block_from_kv(oracle_dims(oracle, w), k, v, pos).serialize()
    assert kvg.kvg_store_export(store.h, bid) == want
