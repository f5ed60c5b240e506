"""Page sizes around the tile heights of the decode kernels and the boxes of the
tensor-copy append: pages smaller than a tile, exact and inexact multiples,
pages copied in several boxes.  Rows written by appends that start and end
inside pages, pool bytes against the oracle; decode over all rows and over
windows that start inside a tile against the fp64 attention."""
import math

import numpy as np
import pytest

import kvg_synth as syn
import oracle as orc
from kvg_testlib import (CANARY, append, compare_decode, decode, dims_for, fill_canary, need_gpu,
                         oracle_dims, pool_u16, tables)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,hkv,g", [(64, 2, 4), (128, 3, 2), (256, 1, 2)])
@pytest.mark.parametrize("page", [1, 3, 15, 16, 17, 32, 48, 58, 59, 64, 65, 100, 128, 300])
def test_append_and_decode(d, hkv, g, page):
    kvg = need_gpu()
    w = syn.Workload("pages", 2, hkv * g, hkv, d, page, 10000.0, 0x80)
    parts = [2 * page + 5, page, 3 * page + 1, 1, page - 1]  # the long ones go by tensor copies
    parts = [n for n in parts if n > 0]
    total = sum(parts)
    n_pages, slots = -(-total // page) + 3, total + page
    c = kvg.Cache(dims_for(kvg, w), n_pages, 2, slots)
    fill_canary(c)
    kvg.kvg_cache_set_free_order(c.h, syn.permutation(n_pages, 81))
    oc = orc.OracleCache(oracle_dims(orc, w), n_pages, 2, slots, fill=CANARY)
    oc.set_free_order(syn.permutation(n_pages, 81))
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, total, 82))
    at = 0
    for n in parts:
        append(kvg, c, 1, k[:, at:at + n], v[:, at:at + n], syn.positions(at, n))
        oc.append(1, k[:, at:at + n], v[:, at:at + n], syn.positions(at, n))
        at += n
    kvg.kvg_sync(c.h)
    assert np.array_equal(pool_u16(c, w), oc.pool)
    pt, pf, ps = tables(c)
    assert np.array_equal(pt, oc.page_table) and np.array_equal(pf, oc.page_fill)
    assert np.array_equal(ps, oc.positions)
    q = syn.as_u16(syn.queries(w, 2, 1, 83))
    scale = 1.0 / math.sqrt(d)
    for windows in ([0, 0], [0, max(1, total - page // 2 - 1)]):
        kvg.kvg_cache_set_layer_windows(c.h, windows)
        oc.set_layer_windows(windows)
        o = decode(kvg, c, w, [1], q)
        for l in range(2):
            compare_decode(orc, o[l, 0], oc.decode(1, l, q[l, 0], scale), what=f"page {page} layer {l}")
    kvg.kvg_sync(c.h)


@pytest.mark.parametrize("page", [4, 16, 24, 32, 33, 48, 64])
def test_fp8_decode(page):
    kvg = need_gpu()
    w = syn.Workload("pages8", 2, 4, 2, 128, page, 10000.0, 0x84)
    n = 5 * page + 3
    ks = vs = syn.FP8_K_SCALE
    dims = kvg.make_dims(2, 2, 128, page, 10000.0, 0, kvg.KVG_KV_E4M3, ks, vs)
    c = kvg.Cache(dims, 7, 1, n)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 85))
    append(kvg, c, 0, k, v, syn.positions(0, n))
    q = syn.as_u16(syn.queries(w, 2, 1, 86))
    o = decode(kvg, c, w, [0], q)
    for l in range(2):
        kk = orc.e4m3_dequant(orc.e4m3_quantize(k[l], ks), ks)
        vv = orc.e4m3_dequant(orc.e4m3_quantize(v[l], vs), vs)
        compare_decode(orc, o[l, 0], orc.gqa_decode_f64kv(q[l, 0], kk, vv, 1.0 / math.sqrt(128)), what=f"page {page}")
    kvg.kvg_sync(c.h)


@pytest.mark.parametrize("d,g", [(128, 1), (128, 4), (256, 2)])
@pytest.mark.parametrize("page", [16, 32, 64])
def test_fp8_decode_rows_outside_are_not_read_as_values(page, d, g):
    """A pool of NaN codes around the rows: a last tile that is partly filled,
    and windows whose first row lies inside a tile."""
    kvg = need_gpu()
    hkv = 1
    w = syn.Workload("nan8", 2, hkv * g, hkv, d, page, 10000.0, 0x87)
    n = 3 * page + 7
    ks = vs = syn.FP8_K_SCALE
    c = kvg.Cache(kvg.make_dims(2, hkv, d, page, 10000.0, 0, kvg.KVG_KV_E4M3, ks, vs), 5, 1, n)
    fill_canary(c)  # 0x7F, the NaN code, in every second byte
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 88))
    append(kvg, c, 0, k, v, syn.positions(0, n))
    q = syn.as_u16(syn.queries(w, 2, 1, 89))
    for first in (0, 5, page + 9):
        kvg.kvg_cache_set_layer_windows(c.h, [0, n - first if first else 0])
        o = decode(kvg, c, w, [0], q)
        for l in range(2):
            lo = first if l == 1 else 0
            kk = orc.e4m3_dequant(orc.e4m3_quantize(k[l][lo:], ks), ks)
            vv = orc.e4m3_dequant(orc.e4m3_quantize(v[l][lo:], vs), vs)
            compare_decode(orc, o[l, 0], orc.gqa_decode_f64kv(q[l, 0], kk, vv, 1.0 / math.sqrt(d)),
                           what=f"page {page} layer {l} from {lo}")
    kvg.kvg_sync(c.h)
