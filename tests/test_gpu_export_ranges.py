"""Exports and imports through 16-byte vectors: every residue of the first recorder and of the destination
against a 16-byte boundary, and counts about a vector, equal the plain slice of the distances."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 7, 8, 9, 17, 40_003])
def test_export_ranges(count):
    import torch
    ctx = ssd.Context(ssd.make_params(dict(log2_eta=8, q=8, r=8, delta=4, k=60, theta=100)), tg.hash_tables(3))
    sk, n = ctx.sketch(), ctx.sketch_bytes // 2
    dist = np.random.default_rng(count).integers(0, 65536, n, dtype=np.uint16)
    dist[::5] = 65535
    dev = torch.from_numpy(dist.view(np.int16)).cuda()
    sk.load_device(dev, 70_000)
    buf = torch.zeros(count + 32, dtype=torch.int16, device="cuda:0")
    for first in list(range(9)) + [n - count]:
        for shift in range(9):
            buf.zero_()
            sk.export_device(buf[shift:shift + count], first, count)
            got = buf.cpu().numpy().view(np.uint16)
            assert np.array_equal(got[shift:shift + count], dist[first:first + count]), (first, shift)
            assert not got[:shift].any() and not got[shift + count:].any(), (first, shift)
    assert np.array_equal(sk.export(), dist)
    ctx.close()
