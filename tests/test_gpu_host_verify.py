"""Verified grafts from a pinned-host store (chunks copied and hashed on the
library's streams) at page and block shapes where the work changes form: pages
of one short leaf, of a whole leaf and a short one, of whole leaves only; one
chunk, a chunk per page, and more pages than chunks.  The pool, the tables and
the report equal the HBM store's graft; a changed byte is found."""
import ctypes

import numpy as np
import pytest
import torch

import kvg_synth as syn
from kvg_testlib import append, dims_for, fill_canary, need_gpu, pool_u16, tables

pytestmark = pytest.mark.gpu


# kv heads, head_dim, page size, layers, tokens
@pytest.mark.parametrize("hkv,d,page,layers,n", [
    (1, 64, 3, 1, 7),        # 384-byte pages, 6 leaves
    (1, 64, 33, 2, 70),      # 4,224-byte pages: a whole leaf and 128 bytes
    (2, 64, 16, 2, 256),     # one whole leaf per page, two groups
    (2, 64, 16, 3, 180),     # a ragged last page, 72 leaves
    (3, 128, 17, 2, 400),    # 13,056-byte pages: three leaves and 768 bytes
    (8, 128, 64, 8, 1300),   # 32-leaf pages, 10,752 leaves: several groups per CTA
    (8, 128, 64, 40, 1300),  # 53,760 leaves: several rounds
])
def test_host_verified_graft(hkv, d, page, layers, n):
    kvg = need_gpu()
    w = syn.Workload("host-verify", layers, hkv, hkv, d, page, 10000.0, 0x65)
    pages = -(-n // page)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 66))
    src = kvg.Cache(dims_for(kvg, w), pages, 1, n)
    append(kvg, src, 0, k, v, syn.positions(5, n))
    out = []
    flags = kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC
    for residency in (kvg.KVG_RESIDENCY_HBM, kvg.KVG_RESIDENCY_PINNED_HOST):
        store = kvg.Store(dims_for(kvg, w), residency, 1 << 30)
        bid = kvg.kvg_deposit(store.h, src.h, 0, 0, n)
        torch.cuda.synchronize()
        c = kvg.Cache(dims_for(kvg, w), pages + 3, 2, n + page)
        fill_canary(c)
        kvg.kvg_cache_set_free_order(c.h, syn.permutation(pages + 3, 67))
        rep = kvg.kvg_graft_report()
        kvg.kvg_graft(store.h, bid, c.h, 1, -1, 0, flags, report=rep)
        assert rep.n_mismatch == 0 and rep.n_pages_checked == 2 * layers * pages
        out.append((pool_u16(c, w), *tables(c)))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    # the last byte of the last plane's first page
    info = kvg.kvg_store_block_info(store.h, bid)
    pb = c.view.page_bytes
    at = info.pages_offset + ((2 * layers - 1) * pages + 1) * pb - 1
    byte = np.frombuffer((ctypes.c_uint8 * 1).from_address(info.bytes + at), np.uint8)
    byte ^= 0x40
    kvg.kvg_cache_release(c.h, 1)
    with pytest.raises(kvg.KvgError) as e:
        kvg.kvg_graft(store.h, bid, c.h, 1, -1, 0, flags, report=rep)
    assert e.value.status == kvg.KVG_ERR_DIGEST
    assert rep.n_mismatch == 1 and rep.mismatch_pages[0] == (2 * layers - 1) * pages


# 64-leaf pages, a page per chunk: 16 leaves per SM (152 SMs) is the most whose chunks are
# hashed in the two-warp form; and chunks of one to three one-leaf pages
@pytest.mark.parametrize("hkv,d,page,layers,n", [(8, 256, 64, 19, 5 * 64), (8, 256, 64, 20, 5 * 64 - 1),
                                                 (2, 64, 16, 2, 32), (2, 64, 16, 3, 700)])
def test_chunked_host_verified_graft(hkv, d, page, layers, n):
    kvg = need_gpu()
    w = syn.Workload("chunked-verify", layers, hkv, hkv, d, page, 10000.0, 0x66)
    pages = -(-n // page)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 67))
    src = kvg.Cache(dims_for(kvg, w), pages, 1, n)
    append(kvg, src, 0, k, v, syn.positions(5, n))
    events = [torch.cuda.Event() for _ in range(16)]
    for e in events:
        e.record()
    out = []
    for residency in (kvg.KVG_RESIDENCY_HBM, kvg.KVG_RESIDENCY_PINNED_HOST):
        store = kvg.Store(dims_for(kvg, w), residency, 1 << 30)
        bid = kvg.kvg_deposit(store.h, src.h, 0, 0, n)
        torch.cuda.synchronize()
        c = kvg.Cache(dims_for(kvg, w), pages + 3, 2, n + page)
        fill_canary(c)
        kvg.kvg_cache_set_free_order(c.h, syn.permutation(pages + 3, 68))
        rep = kvg.kvg_graft_report()
        ends = kvg.kvg_graft_chunked(store.h, bid, c.h, 1, [e.cuda_event for e in events], -1, 0,
                                     kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC, report=rep)
        assert ends[-1] == n and rep.n_mismatch == 0 and rep.n_pages_checked == 2 * layers * pages
        out.append((pool_u16(c, w), *tables(c)))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    info = kvg.kvg_store_block_info(store.h, bid)
    byte = np.frombuffer((ctypes.c_uint8 * 1).from_address(info.bytes + info.pages_offset), np.uint8)
    byte ^= 1
    kvg.kvg_cache_release(c.h, 1)
    with pytest.raises(kvg.KvgError) as e:
        kvg.kvg_graft_chunked(store.h, bid, c.h, 1, [e.cuda_event for e in events], -1, 0,
                              kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC, report=rep)
    assert e.value.status == kvg.KVG_ERR_DIGEST and rep.n_mismatch == 1 and rep.mismatch_pages[0] == 0
