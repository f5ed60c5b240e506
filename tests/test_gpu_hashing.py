"""Digests at the sizes where the two-warp hashing changes course: message
tails around the padding's block boundaries (odd and even block counts, since
blocks are handed over in pairs), and pages whose count and leaf count leave
lanes or half a pair empty."""
import hashlib

import numpy as np
import pytest
import torch

from kvg_testlib import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 4, 55, 56, 59, 60, 63, 64, 65, 119, 120, 128, 183, 184, 192, 4096, 4160, 5000])
@pytest.mark.parametrize("at", [0, 4, 3])
def test_plain_digest_tails(n, at):
    kvg = need_gpu()
    data = np.random.default_rng(n).integers(0, 256, n + 8, dtype=np.uint8)
    buf = torch.from_numpy(data).cuda()
    out = torch.zeros(32, dtype=torch.uint8, device="cuda")
    kvg.kvg_digest(buf.data_ptr() + at, n, kvg.KVG_SHA256_PLAIN, 0, out.data_ptr())
    torch.cuda.synchronize()
    assert bytes(out.cpu().numpy()) == hashlib.sha256(data[at:at + n].tobytes()).digest()


@pytest.mark.parametrize("leaves", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("pages", [1, 15, 16, 17, 33])
def test_page_digest_counts(oracle, leaves, pages):
    kvg = need_gpu()
    pb = 4096 * leaves
    data = np.random.default_rng(leaves * 100 + pages).integers(0, 256, pages * pb, dtype=np.uint8)
    buf = torch.from_numpy(data).cuda()
    out = torch.zeros(32 * pages, dtype=torch.uint8, device="cuda")
    kvg.kvg_digest(buf.data_ptr(), data.size, kvg.KVG_SHA256_PAGED, pb, out.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().reshape(pages, 32), oracle.page_digests(data, pb))
