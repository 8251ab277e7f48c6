"""The one-router slot's touch lists for every relation of chunks to rows (eight, four, two chunks per row, one,
two rows per chunk, one chunk in all), slots about a warp and a block of pairs, buffers that start at 8
mod 16 bytes, and both sides and an IP group: the list and every recorder equal scan + close_slot."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg
from gpu_harness import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [64 << 10, 128 << 10, 256 << 10, 512 << 10, 1 << 20, 4 << 20])
@pytest.mark.parametrize("view", [(0, 0, 0), (1, 0, 0), (0, 2, 1)])
def test_list_chunks(chunk, view):
    prm = dict(log2_eta=8, q=14, r=5, delta=6, k=3, theta=60)
    tabs = tg.hash_tables(9)
    rng = np.random.default_rng(chunk + view[0] + 7 * view[1])
    a = ssd.Context(ssd.make_params(prm, touch_chunk_bytes=chunk), tabs)
    b = ssd.Context(ssd.make_params(prm), tabs)
    ra, rb = a.sketch().set_view(*view), b.sketch().set_view(*view)
    found = 0
    for n, skip in [(0, 0), (1, 0), (1, 1), (2, 1), (63, 0), (64, 1), (65, 1), (513, 0), (4098, 1), (60_001, 1)]:
        hosts = rng.integers(0, 1 << 32, 40, dtype=np.uint64).astype(np.uint32)
        pairs = np.empty((n + skip, 2), dtype=np.uint32)
        pairs[:, view[0]] = hosts[rng.integers(0, 40, n + skip)]
        pairs[:, 1 - view[0]] = rng.integers(0, 1 << 32, n + skip, dtype=np.uint64)
        dev = to_dev(pairs)[2 * skip:]     # starts at 8 mod 16 bytes
        b.scan(rb, dev)
        want = b.close_slot([rb])
        got = a.slot([ra], [dev])
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), (n, skip)
        assert np.array_equal(ra.export(), rb.export()), (n, skip)
        found += len(want[0])
    assert found > 0
    a.close()
    b.close()
