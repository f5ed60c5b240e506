"""Verified batches of grafts: the pages restored and the mismatches found are
those of the same grafts one at a time, for own-position and re-based grafts,
from HBM and pinned host memory, for launches of each hashing form, and where
the leaf digests are worked off in slices."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import kvg_synth as syn
from kvg_testlib import append, dev_view, dims_for, fill_canary, geometry, need_gpu, pool_u16, tables

pytestmark = pytest.mark.gpu


def _library(kvg, w, lens, residency):
    P = w.page_size
    src = kvg.Cache(dims_for(kvg, w), max(-(-n // P) for n in lens), 1, max(lens))
    store = kvg.Store(dims_for(kvg, w), residency, 2 << 30)
    bids = []
    for i, n in enumerate(lens):
        k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 300 + i))
        append(kvg, src, 0, k, v, syn.positions(0, n))
        bids.append(kvg.kvg_deposit(store.h, src.h, 0, 0, n))
        kvg.kvg_cache_release(src.h, 0)
    torch.cuda.synchronize()
    return store, bids


def _caches(kvg, w, lens, seqs, n):
    P = w.page_size
    out = []
    for _ in range(n):
        c = kvg.Cache(dims_for(kvg, w), sum(-(-x // P) for x in lens) + 1, max(seqs) + 1, sum(lens) + P * len(lens))
        fill_canary(c)
        out.append(c)
    return out


def _flip(addr, residency):
    byte = dev_view(addr, 1) if residency == 0 else np.frombuffer((ctypes.c_uint8 * 1).from_address(addr), np.uint8)
    byte ^= 1
    torch.cuda.synchronize()


# blocks of 70, 1 and 33 pages of one 4 KiB leaf (two-warp form), and enough
# 64-leaf pages for the one-warp forms: the register form, and a full wave
@pytest.mark.parametrize("geo,layers,lens", [("tiny", 2, [70 * 16, 5, 33 * 16 - 3]),
                                             ("d128", 3, [6 * 64, 2 * 64 + 5, 9 * 64]),
                                             ("d128", 24, [16 * 64, 64, 9 * 64 - 1])])
@pytest.mark.parametrize("deltas", [None, [0, 70, 0]])
@pytest.mark.parametrize("residency", [0, 1])
def test_verified_batch_equals_single_grafts(geo, layers, lens, deltas, residency):
    kvg = need_gpu()
    w = geometry(geo).with_layers(layers)
    store, bids = _library(kvg, w, lens, residency)
    seqs = [1, 0, 1]
    one, batch = _caches(kvg, w, lens, seqs, 2)
    flags = kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC
    for i in range(3):
        kvg.kvg_graft(store.h, bids[i], one.h, seqs[i], -1, deltas[i] if deltas else 0, flags)
    rep = kvg.kvg_graft_report()
    kvg.kvg_graft_batch(store.h, bids, batch.h, seqs, flags, report=rep, deltas=deltas)
    assert rep.n_mismatch == 0 and rep.n_pages_checked == 2 * layers * sum(-(-n // w.page_size) for n in lens)
    assert np.array_equal(pool_u16(one, w), pool_u16(batch, w))
    for a, b in zip(tables(one), tables(batch)):
        assert np.array_equal(a, b)
    # the last graft's block with a byte changed, not waited for; then, mended,
    # the middle one's: both pages are listed, under the later batch's sequence
    pages = []
    for victim, plane in ((2, 1), (1, 0)):
        npb = -(-lens[victim] // w.page_size)
        pages.append(plane * npb + npb - 1)
        info = kvg.kvg_store_block_info(store.h, bids[victim])
        at = info.bytes + info.pages_offset + pages[-1] * batch.view.page_bytes + 3
        _flip(at, residency)
        for sq in (0, 1):
            kvg.kvg_cache_release(batch.h, sq)
        if victim == 2:
            kvg.kvg_graft_batch(store.h, bids, batch.h, seqs, kvg.KVG_GRAFT_VERIFY, deltas=deltas)
            torch.cuda.synchronize()
            _flip(at, residency)
    with pytest.raises(kvg.KvgError) as e:
        kvg.kvg_graft_batch(store.h, bids, batch.h, seqs, flags, report=rep, deltas=deltas)
    assert e.value.status == kvg.KVG_ERR_DIGEST
    assert rep.seq == seqs[1] and rep.n_mismatch == 2
    assert sorted(rep.mismatch_pages[:2]) == sorted(pages)
    kvg.kvg_sync(batch.h)


_CHILD = """
import sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import test_gpu_batch_verify as t
t.slices()
"""


def slices():
    """Four blocks of 1,000 one-leaf pages in 16 planes: 64,000 leaves, two slices of 1 MiB of leaf digests."""
    kvg = need_gpu()
    w = geometry("tiny").with_layers(8)
    lens = [16 * 1000] * 4
    store, bids = _library(kvg, w, lens, 0)
    one, batch = _caches(kvg, w, lens, [0, 1], 2)
    seqs = [0, 1, 0, 1]
    kvg.kvg_graft_batch(store.h, bids, one.h, seqs, 0)
    rep = kvg.kvg_graft_report()
    flags = kvg.KVG_GRAFT_VERIFY | kvg.KVG_GRAFT_SYNC
    kvg.kvg_graft_batch(store.h, bids, batch.h, seqs, flags, report=rep)
    assert rep.n_mismatch == 0
    assert np.array_equal(pool_u16(one, w), pool_u16(batch, w))
    for a, b in zip(tables(one), tables(batch)):
        assert np.array_equal(a, b)
    info = kvg.kvg_store_block_info(store.h, bids[3])
    byte = dev_view(info.bytes + info.pages_offset + (5 * 1000 + 999) * batch.view.page_bytes, 1)
    byte ^= 1
    for s in (0, 1):
        kvg.kvg_cache_release(batch.h, s)
    try:
        kvg.kvg_graft_batch(store.h, bids, batch.h, seqs, flags, report=rep)
        raise AssertionError("mismatch not reported")
    except kvg.KvgError as e:
        assert e.status == kvg.KVG_ERR_DIGEST
    assert rep.seq == 1 and rep.n_mismatch == 1 and rep.mismatch_pages[0] == 5999


def test_verified_batch_in_slices():
    need_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _CHILD, root], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, KVG_BATCH_LEAF_MB="1"))
    assert r.returncode == 0, r.stderr[-2000:]
