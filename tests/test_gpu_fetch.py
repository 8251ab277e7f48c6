"""Lists fetched with sync=True equal the device outputs of the same slot: an empty list, a short one and one
longer than the part that is copied ahead, into default and into given buffers of either 4-byte type."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg
from gpu_harness import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hosts", [0, 3, 4600])
def test_fetched_lists(hosts):
    import torch
    # theta = 1: every touched estimator is hot, so every host is listed
    prm = dict(log2_eta=5, q=14, r=5, delta=6, k=1, theta=1)
    ctx = ssd.Context(ssd.make_params(prm, ssd.SSD_VERIFY_H0), tg.hash_tables(4))
    rng = np.random.default_rng(hosts)
    pairs = to_dev(rng.integers(0, 1 << 32, (hosts, 2), dtype=np.uint64).astype(np.uint32))
    cap = 1 << 16
    dev = (torch.zeros(cap, dtype=torch.int32, device="cuda:0"), torch.zeros(cap, dtype=torch.int32, device="cuda:0"),
           torch.zeros(1, dtype=torch.int64, device="cuda:0"))
    ctx.slot([ctx.sketch()], [pairs], out=dev, sync=False)
    torch.cuda.synchronize()
    m = int(dev[2].item())
    assert m >= hosts - 1 and (hosts < 4600 or m > ctx._HEAD)
    want = [x[:m].cpu().numpy().view(np.uint32) for x in dev[:2]]
    outs = [None, tuple(torch.empty_like(x) for x in dev),
            (torch.empty(cap, dtype=torch.float32, device="cuda:0"), torch.empty(cap, dtype=torch.float32, device="cuda:0"),
             torch.empty_like(dev[2]))]
    for out in outs:
        got = ctx.slot([ctx.sketch()], [pairs], out=out)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    ctx.close()
