"""Copies that take several small pages at a time (graft, re-based graft, batch,
deposit): page counts that fill units, leave a short last unit and a ragged
last page, and ones that take a page at a time, from HBM and pinned host
memory, against the oracle; re-based keys within the rounding of the rotation."""
import numpy as np
import pytest
import torch

import kvg_synth as syn
import oracle as orc
from kvg_testlib import (CANARY, append, check_rotation_rounding, dims_for, fill_canary, need_gpu, oracle_dims, pool_u16,
                         tables)

pytestmark = pytest.mark.gpu


def rotated(k, delta, theta, style):
    """Key rows [..., D] (bf16 bits) moved by delta positions, in fp64 (style 0: pairs i, i + D/2; 1: 2i, 2i + 1)."""
    x = orc.bf16_to_f64(k)
    d = x.shape[-1]
    angle = delta * theta ** (-2.0 * np.arange(d // 2) / d)
    at = (slice(0, d // 2), slice(d // 2, d)) if style == 0 else (slice(0, d, 2), slice(1, d, 2))
    a, b = x[..., at[0]], x[..., at[1]]
    out = np.empty_like(x)
    out[..., at[0]] = a * np.cos(angle) - b * np.sin(angle)
    out[..., at[1]] = a * np.sin(angle) + b * np.cos(angle)
    return out


# 4 KiB pages in 2 x 16 planes: from 4 x 152 pages a unit has two, from 16 x 4 x 152 sixteen
@pytest.mark.parametrize("pages,ragged", [(18, 3), (40, 0), (57, 5), (304, 1), (700, 0), (701, 15)])
@pytest.mark.parametrize("style", [0, 1])
@pytest.mark.parametrize("residency", [0, 1])
def test_units_of_several_pages(pages, ragged, style, residency):
    kvg = need_gpu()
    w = syn.Workload("small", 16, 2, 2, 64, 16, 10000.0, 0x90)
    n = pages * 16 - ragged
    dims = dims_for(kvg, w, style)
    od = oracle_dims(orc, w, style)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 91))
    pos = syn.positions(0, n)
    src = kvg.Cache(dims, pages, 1, n)
    kvg.kvg_cache_set_free_order(src.h, syn.permutation(pages, 92))
    append(kvg, src, 0, k, v, pos)
    store = kvg.Store(dims, residency, 1 << 30)
    bid = kvg.kvg_deposit(store.h, src.h, 0, 0, n)
    blk = orc.block_from_kv(od, k, v, pos)
    assert kvg.kvg_store_export(store.h, bid) == blk.serialize()
    k64 = rotated(k, 4097, w.rope_theta, style)
    assert np.allclose(k64[0, 0], orc.rope_rotate_rows(k[0, 0], 4097, w.rope_theta, style), rtol=0, atol=1e-11)
    # own position; re-based; a batch of both
    cp = 2 * pages + 5
    slots = 2 * pages * 16
    for how in ("graft", "batch"):
        c = kvg.Cache(dims, cp, 2, slots)
        fill_canary(c)
        kvg.kvg_cache_set_free_order(c.h, syn.permutation(cp, 93))
        oc = orc.OracleCache(od, cp, 2, slots, fill=CANARY)
        oc.set_free_order(syn.permutation(cp, 93))
        if how == "graft":
            kvg.kvg_graft(store.h, bid, c.h, 0, -1, 0, 0)
            kvg.kvg_graft(store.h, bid, c.h, 1, -1, 4097, 0)
        else:
            kvg.kvg_graft_batch(store.h, [bid, bid], c.h, [0, 1], 0, deltas=[0, 4097])
        oc.graft(0, blk)
        oc.graft(1, blk, delta=4097)
        torch.cuda.synchronize()
        got, want = pool_u16(c, w), oc.pool
        pt, pf, ps = tables(c)
        assert np.array_equal(pt, oc.page_table) and np.array_equal(pf, oc.page_fill)
        assert np.array_equal(ps, oc.positions)
        moved = pt[1][pt[1] >= 0]
        keys = np.zeros(cp, bool)
        keys[moved] = True
        assert np.array_equal(got[:, 1], want[:, 1]) and np.array_equal(got[:, 0, ~keys], want[:, 0, ~keys])
        # re-based keys: every valid row within the fp32 rotation's rounding of the
        # fp64 one, padding rows untouched
        logical = [np.swapaxes(x[:, 0, moved], 2, 3).reshape(w.n_layers, pages * 16, 2, 64) for x in (got, want)]
        check_rotation_rounding(orc, logical[0][:, :n], k64)
        assert np.array_equal(logical[0][:, n:], logical[1][:, n:])
        if how == "graft":
            single = got
        else:
            assert np.array_equal(got, single)
        kvg.kvg_sync(c.h)


@pytest.mark.parametrize("verify", [0, 1])
@pytest.mark.parametrize("style", [0, 1])
@pytest.mark.parametrize("residency", [0, 1])
def test_batch_of_own_and_rebased_pages_in_turn(verify, style, residency):
    """Units of a batch that hold runs of own-position and of re-based pages, against a graft at a time."""
    kvg = need_gpu()
    w = syn.Workload("runs", 16, 2, 2, 64, 16, 10000.0, 0x91)
    lens = [3 * 16, 18 * 16 - 5, 7, 40 * 16, 16, 29 * 16 - 1]
    deltas = [0, 9, 0, 4097, 9, 0]
    dims = dims_for(kvg, w, style)
    src = kvg.Cache(dims, 40, 1, 640)
    store = kvg.Store(dims, residency, 1 << 30)
    bids = []
    for i, n in enumerate(lens):
        k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 94 + i))
        append(kvg, src, 0, k, v, syn.positions(0, n))
        bids.append(kvg.kvg_deposit(store.h, src.h, 0, 0, n))
        kvg.kvg_cache_release(src.h, 0)
    torch.cuda.synchronize()
    times = 6  # 558 pages in 2 x 16 planes: sixteen to a unit
    pages = times * sum(-(-n // 16) for n in lens)
    seqs = [i // len(lens) for i in range(times * len(lens))]
    flags = kvg.KVG_GRAFT_VERIFY if verify else 0
    got = []
    for how in ("batch", "single"):
        c = kvg.Cache(dims, pages + 3, times, pages * 16)
        fill_canary(c)
        kvg.kvg_cache_set_free_order(c.h, syn.permutation(pages + 3, 95))
        if how == "batch":
            kvg.kvg_graft_batch(store.h, bids * times, c.h, seqs, flags, deltas=deltas * times)
        else:
            for b, s, d in zip(bids * times, seqs, deltas * times):
                kvg.kvg_graft(store.h, b, c.h, s, -1, d, flags)
        torch.cuda.synchronize()
        kvg.kvg_sync(c.h)
        got.append((pool_u16(c, w), *tables(c)))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
