"""Merge of the split-K partials against the CPU oracle at the partial counts
where its work split changes: one partial, one lane group's loads, several
groups, more partials than a block's groups take in one round, and the most a
head can have (every resident warp on one kv head), for each head_dim and both
outputs (bf16, and the split decode's state)."""
import math

import pytest
import torch

import kvg_synth as syn
from kvg_testlib import append, compare_decode, dims_for, need_gpu, to_dev, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,g", [(64, 4), (128, 2), (256, 2)])
@pytest.mark.parametrize("tiles", [1, 2, 3, 9, 33, 130, 700])
def test_combine_partial_counts(oracle, d, g, tiles):
    kvg = need_gpu()
    tok = {64: 64, 128: 64, 256: 16}[d]  # rows of a decode tile
    n = tiles * tok - 5
    w = syn.Workload("one-head", 1, g, 1, d, 64, 10000.0, 0x60)
    pages = -(-n // w.page_size)
    c = kvg.Cache(dims_for(kvg, w), pages + 1, 2, (pages + 1) * w.page_size)
    k, v = (syn.as_u16(x) for x in syn.kv_rows(w, n, 61 + tiles))
    append(kvg, c, 0, k, v, syn.positions(0, n))
    q = syn.as_u16(syn.queries(w, 1, 1, 62))
    qd = to_dev(q)
    out, out2 = torch.empty_like(qd), torch.empty_like(qd)
    state = torch.full((1, 1, g, d + 4), float("nan"), dtype=torch.float32, device="cuda")
    scale = 1.0 / math.sqrt(d)
    kvg.kvg_decode_attention(c.h, 0, [0], qd.data_ptr(), g, out.data_ptr(), scale)
    kvg.kvg_decode_attention_range(c.h, 0, [0], qd.data_ptr(), g, scale, 0, (pages + 1) * w.page_size, 0,
                                   state.data_ptr())
    kvg.kvg_decode_state_finish(state.data_ptr(), g, d, out2.data_ptr())
    kvg.kvg_sync(c.h)
    ref = oracle.gqa_decode(q[0, 0], k[0], v[0], scale)
    compare_decode(oracle, u16(out)[0, 0], ref)
    compare_decode(oracle, u16(out2)[0, 0], ref)
