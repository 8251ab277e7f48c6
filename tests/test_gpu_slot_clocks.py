"""A slot whose touches are applied by the streaming pass against the same slot scanned and closed, for several
routers at one clock and at differing ones: equal lists, merged sketches and recorders. The recorders include
stamps older than the clocks' last wrap, never set ones and ones about to reach 65535, beside the
slot's own touches, and the clocks those at which stamps wrap."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg
from gpu_harness import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots,group", [((40, 65534, 700), 8), ((65534,) * 3, 4), ((65535 + 3,) * 9, 8), ((9, 65535 + 9), 4),
                                         ((100, 100), 8), ((100, 101, 102, 103, 104), 2), ((65535 + 3,) * 3, 2)])
@pytest.mark.parametrize("log2_eta", [6, 8, 11])
def test_slot_equals_scan_and_close(slots, log2_eta, group):
    eta, q, r, k, n = 1 << log2_eta, 8, 8, 60, len(slots)
    rng = np.random.default_rng(log2_eta * 100 + n)
    flags, prm = ssd.SSD_SLOT_CHUNKED, dict(log2_eta=log2_eta, q=q, r=r, delta=4, k=k, theta=eta // 2)
    kinds = np.array([0, k - 1, k, 20000, 65500, 65533, 65534, 65535], dtype=np.uint16)
    images = [rng.choice(kinds, r * (eta << q), p=[.005, .005, .1, .2, .1, .1, .1, .39]) for _ in range(n)]
    pairs = []
    for j in range(n):   # sparse sources, and two hosts whose peers fill their estimators
        p = rng.integers(0, 1 << 32, (4 * eta + 2 * eta + 37 * j, 2), dtype=np.uint64).astype(np.uint32)
        p[:2 * eta, 0] = np.repeat(np.array([0x0A000001, 0xC0A80102], dtype=np.uint32), eta)
        pairs.append(p)
    got = []
    for fused in (True, False):
        ctx = ssd.Context(ssd.make_params(prm, flags), tg.hash_tables(3))
        ctx.tuning = dict(merge_group=group)
        routers, merged = [ctx.sketch() for _ in range(n)], ctx.sketch()
        for sk, image, slot in zip(routers, images, slots):
            sk.load(image, slot)
            sk.slot = slots[0]
        dev = [to_dev(p) for p in pairs]
        if fused:
            lists = ctx.slot(routers, dev, merged)
        else:
            ctx.scan_batch(routers, dev)
            lists = ctx.close_slot(routers, merged)
        got.append([*lists, merged.export(), *(sk.export() for sk in routers), np.array(ctx.stats()["hot"])])
        ctx.close()
    assert len(got[0][0]) >= 1
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    # the merged sketch is the least distance of the scanned routers, which are each advanced by one
    before = [np.where(x == 65535, x, x - 1) for x in got[0][3:3 + n]]
    known = np.minimum.reduce([np.where((x == 65535) & (im == 65534), np.uint16(65534), x) for x, im in zip(before, images)])
    assert np.array_equal(got[0][2], known)
