"""Decode over layers with different windows: one, two, three and five window
sizes in a call (one launch takes two), first groups that read nothing and
batches that do not fit one launch, against the oracle; the allocation-free
entry point gives the same bytes."""
import math

import numpy as np
import pytest
import torch

import kvg_synth as syn
import oracle as orc
from kvg_testlib import append, compare_decode, decode, dims_for, need_gpu, oracle_dims, to_dev, u16

pytestmark = pytest.mark.gpu

LENS = [1, 70, 0, 333, 128]


@pytest.mark.parametrize("windows", [[0] * 6, [48] * 6, [0, 17, 0, 17, 17, 0], [33, 0, 33, 100, 0, 100],
                                     [1, 0, 64, 200, 9, 0]])
@pytest.mark.parametrize("d,g,page", [(64, 2, 16), (128, 4, 64), (256, 2, 24)])
def test_windows_of_several_sizes(windows, d, g, page):
    kvg = need_gpu()
    w = syn.Workload("groups", 6, 2 * g, 2, d, page, 10000.0, 0x70)
    n_pages, slots = sum(-(-n // page) for n in LENS) + 2, 400
    c = kvg.Cache(dims_for(kvg, w), n_pages, len(LENS), slots)
    oc = orc.OracleCache(oracle_dims(orc, w), n_pages, len(LENS), slots)
    for i, n in enumerate(LENS):
        if n:
            k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 71 + i))
            append(kvg, c, i, k, v, syn.positions(0, n))
            oc.append(i, k, v, syn.positions(0, n))
    kvg.kvg_cache_set_layer_windows(c.h, windows)
    oc.set_layer_windows(windows)
    order = [3, 0, 4, 2, 1]
    q = syn.as_u16(syn.queries(w, w.n_layers, len(order), 72))
    o = decode(kvg, c, w, order, q)
    scale = 1.0 / math.sqrt(d)
    for l in range(w.n_layers):
        for b, sq in enumerate(order):
            if LENS[sq]:
                compare_decode(orc, o[l, b], oc.decode(sq, l, q[l, b], scale), what=f"layer {l} seq {sq}")
            else:
                assert not o[l, b].any()
    qd = to_dev(q)
    out = torch.empty_like(qd)
    kvg.kvg_decode_attention_noalloc(c.h, -1, order, qd.data_ptr(), w.n_q_heads, out.data_ptr(), scale)
    torch.cuda.synchronize()
    assert np.array_equal(u16(out), o)
    # only the sequences of one row and none: the windowed layers read as much as the others
    o2 = decode(kvg, c, w, [2, 0], np.ascontiguousarray(q[:, :2]))
    assert not o2[:, 0].any() and o2[:, 1].any()


@pytest.mark.parametrize("d,g,page,fp8", [(128, 2, 64, True), (256, 2, 64, True), (128, 4, 64, False),
                                          (64, 2, 16, False)])
def test_sharing_a_launch_keeps_the_reduction(d, g, page, fp8):
    """A layer gives the same bytes whether or not another window's layers run in the call."""
    kvg = need_gpu()
    w = syn.Workload("share", 4, 4 * g, 4, d, page, 10000.0, 0x73)
    batch, n, window = 12, 1500, 700
    pages = -(-n // page)
    rows = [[to_dev(syn.as_u16(x)) for x in syn.kv_rows(w, n, 74 + i)] for i in range(batch)]
    pos = to_dev(syn.positions(0, n).astype(np.int32))

    def run(layers, windows):
        dims = kvg.make_dims(len(layers), w.n_kv_heads, d, page, w.rope_theta, 0,
                             kvg.KVG_KV_E4M3 if fp8 else kvg.KVG_KV_BF16, 0.0625, 0.0625)
        c = kvg.Cache(dims, batch * pages, batch, n)
        for i, (k, v) in enumerate(rows):
            kk, vv = k[layers].contiguous(), v[layers].contiguous()
            kvg.kvg_cache_append(c.h, i, kk.data_ptr(), vv.data_ptr(), pos.data_ptr(), n)
            torch.cuda.synchronize()
        kvg.kvg_cache_set_layer_windows(c.h, windows)
        qd = to_dev(q[layers])
        out = torch.empty_like(qd)
        kvg.kvg_decode_attention(c.h, -1, list(range(batch)), qd.data_ptr(), w.n_q_heads, out.data_ptr(),
                                 1.0 / math.sqrt(d))
        torch.cuda.synchronize()
        return u16(out)

    q = syn.as_u16(syn.queries(w, w.n_layers, batch, 75))
    together = run([0, 1, 2, 3], [window, 0, window, 0])
    assert np.array_equal(together[[1, 3]], run([1, 3], [0, 0]))
    assert np.array_equal(together[[0, 2]], run([0, 2], [window, window]))
