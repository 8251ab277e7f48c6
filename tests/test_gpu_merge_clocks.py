"""The streaming passes over several routers against elementwise numpy on the distances: merge, merged
recorders below k per estimator, and advance, at clocks where stamps wrap (slot counter modulo 65535
near 0, below k and at 65534), with recorders that are fresh, inside and outside the window, about to
reach 65535 and never set, and with routers whose clocks differ. Router counts cover every split of the
loads (2, up to 4, 8 and more). Everything is integer arithmetic: results are equal, not close."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg

pytestmark = pytest.mark.gpu


def distances(rng, r, cols, eta, k, dense):
    """Random recorders: mostly old or never, `dense` columns of each row mostly inside the window."""
    kind = rng.random((r, cols, eta), dtype=np.float32)
    d = np.full((r, cols, eta), 65535, dtype=np.uint16)
    old = kind < 0.5
    # (under a window of nearly every distance they lie outside it, or every estimator would be hot)
    d[old] = rng.integers(k if k > 1000 else 0, 65535, int(old.sum()), dtype=np.uint16)
    edge = (kind >= 0.5) & (kind < 0.55)
    d[edge] = rng.choice(np.array([0, k - 1, k, 65533, 65534], dtype=np.uint16), int(edge.sum()))
    for row in range(r):
        for c in dense:
            some = rng.random(eta) < 0.5
            d[row, c, some] = rng.integers(0, k, int(some.sum()), dtype=np.uint16)
    return d


def advanced(d):
    return np.where(d < 65535, d + np.uint16(1), d)


@pytest.mark.parametrize("n,log2_eta,k,slots", [
    (1, 11, 60, (5,)), (2, 8, 60, (5, 5)), (2, 10, 300, (299, 299)), (2, 11, 1, (65534, 65534)),
    (3, 9, 60, (65535, 65535, 65535)), (4, 11, 65534, (7, 7, 7, 7)), (4, 8, 60, (58, 58, 58, 58)),
    (5, 9, 60, (1000,) * 5), (9, 10, 17, (65536,) * 9), (3, 10, 60, (40, 65534, 700)), (2, 9, 300, (100, 101))])
@pytest.mark.parametrize("group", [2, 4, 8])
def test_streaming_passes_equal_numpy(n, log2_eta, k, slots, group):
    import torch
    eta, q, r = 1 << log2_eta, 8, 8
    rng = np.random.default_rng(log2_eta * 1000 + n * 10 + k)
    ctx = ssd.Context(ssd.make_params(dict(log2_eta=log2_eta, q=q, r=r, delta=4, k=k, theta=eta // 2)), tg.hash_tables(3))
    ctx.tuning = dict(merge_group=group)
    routers = [ctx.sketch() for _ in range(n)]
    merged, single = ctx.sketch(), ctx.sketch()
    dist = [distances(rng, r, 1 << q, eta, k, (3, 77, 200)) for _ in range(n)]
    for sk, d, slot in zip(routers, dist, slots):
        sk.load(d.reshape(-1), slot)
        sk.slot = slots[0]     # the host's counters agree; the device clocks are those of the loads
    want = np.minimum.reduce(dist)

    def check_close(first):
        ips, rk = ctx.close_slot(routers, merged if first else None)
        hot = ((want < k).sum(axis=2) >= ctx.threshold).sum(axis=1)
        assert ctx.stats()["hot"] == list(hot)
        single.load(want.reshape(-1), slots[0])
        ref = ctx.regain(single)
        assert np.array_equal(ips, ref[0]) and np.array_equal(rk, ref[1])

    ctx.merge(routers, merged)
    assert np.array_equal(merged.export(), want.reshape(-1))
    check_close(True)
    assert np.array_equal(merged.export(), want.reshape(-1))
    dist = [advanced(d) for d in dist]
    for sk, d in zip(routers, dist):
        assert np.array_equal(sk.export(), d.reshape(-1))
    want = np.minimum.reduce(dist)
    check_close(False)
    dist = [advanced(d) for d in dist]
    ctx.advance(routers)
    for sk, d in zip(routers, dist):
        assert np.array_equal(sk.export(), advanced(d).reshape(-1))
    torch.cuda.synchronize()
    ctx.close()
