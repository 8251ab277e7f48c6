"""Exports and imports whose two ends lie differently against a 16-byte boundary: counts about one and two vectors at
every pair of residues, and the time of a large one against that of an aligned one (the same bytes; one
recorder at a time it took 4.8 times as long, the bound is 2)."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [2, 15, 16, 23, 24, 25, 31, 33])
def test_counts_about_the_vectors(count):
    import torch
    ctx = ssd.Context(ssd.make_params(dict(log2_eta=8, q=8, r=8, delta=4, k=60, theta=100)), tg.hash_tables(3))
    sk, n = ctx.sketch(), ctx.sketch_bytes // 2
    dist = np.random.default_rng(count).integers(0, 65536, n, dtype=np.uint16)
    sk.load(dist, 70_000)
    buf = torch.zeros(count + 32, dtype=torch.int16, device="cuda:0")
    for first in [*range(8), n - count - 3, n - count]:
        for shift in range(8):
            buf.zero_()
            sk.export_device(buf[shift:shift + count], first, count)
            got = buf.cpu().numpy().view(np.uint16)
            assert np.array_equal(got[shift:shift + count], dist[first:first + count]), (first, shift)
            assert not got[:shift].any() and not got[shift + count:].any(), (first, shift)
    for shift in range(1, 8):
        src = torch.zeros(n + 8, dtype=torch.int16, device="cuda:0")
        src[shift:shift + n] = torch.from_numpy(np.roll(dist, shift).view(np.int16)).cuda()
        sk.load_device(src[shift:shift + n], 5)
        assert np.array_equal(sk.export(), np.roll(dist, shift)), shift
    ctx.close()


def test_time_of_a_shifted_export():
    import torch
    ctx = ssd.Context(ssd.make_params(dict(log2_eta=11, q=16, r=5, delta=6, k=60, theta=1024)), tg.hash_tables(3))
    sk, count = ctx.sketch(), ctx.sketch_bytes // 2 - 64
    buf = torch.empty(count + 64, dtype=torch.int16, device="cuda:0")

    def us(first, shift):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sk.export_device(buf[shift:shift + count], first, count)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[3]

    us(0, 0)
    for first, shift in ((1, 0), (0, 3), (4, 0), (8, 1)):
        assert us(first, shift) < 2 * us(0, 0)
    ctx.close()
