"""Lists fetched with sync=True into every kind of output buffer a call takes: pinned host memory that the device
writes, a length of another shape, two-dimensional lists; and with the staging made under inference mode or
another default device. The lists are those of the default buffers."""
import numpy as np
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg
from gpu_harness import to_dev

pytestmark = pytest.mark.gpu
CAP, HOSTS = 1 << 14, 3000


@pytest.fixture
def case():
    # theta = 1: every touched estimator is hot, so every host is listed
    ctx = ssd.Context(ssd.make_params(dict(log2_eta=5, q=14, r=5, delta=6, k=1, theta=1), ssd.SSD_VERIFY_H0),
                      tg.hash_tables(4))
    rng = np.random.default_rng(3)
    pairs = to_dev(rng.integers(0, 1 << 32, (HOSTS, 2), dtype=np.uint64).astype(np.uint32))
    yield ctx, lambda out=None: ctx.slot([ctx.sketch()], [pairs], out=out)
    ctx.close()


def want(ctx, slot):
    """The list by the call's device outputs, not by the fetched ones."""
    import torch
    dev = (torch.zeros(CAP, dtype=torch.int32, device=ctx.device), torch.zeros(CAP, dtype=torch.int32, device=ctx.device),
           torch.zeros(1, dtype=torch.int64, device=ctx.device))
    slot(dev)
    torch.cuda.synchronize()
    m = int(dev[2])
    assert m >= HOSTS - 1
    return [x[:m].cpu().numpy().view(np.uint32) for x in dev[:2]]


def same(got, ref):
    assert np.array_equal(got[0].reshape(-1), ref[0]) and np.array_equal(got[1].reshape(-1), ref[1])


@pytest.mark.parametrize("lists,length", [("pinned", "pinned"), ("pinned", "device"), ("device", "pinned"),
                                          ("device", "1 x 1"), ("device", "scalar"), ("column", "device")])
def test_output_buffers(case, lists, length):
    import torch
    ctx, slot = case
    ref = want(ctx, slot)
    rows = [torch.zeros(CAP, dtype=torch.int32, pin_memory=True) if lists == "pinned" else
            torch.zeros((CAP, 1) if lists == "column" else CAP, dtype=torch.int32, device=ctx.device) for _ in range(2)]
    n_out = (torch.zeros(1, dtype=torch.int64, pin_memory=True) if length == "pinned" else
             torch.zeros({"1 x 1": (1, 1), "scalar": ()}.get(length, (1,)), dtype=torch.int64, device=ctx.device))
    same(slot((*rows, n_out)), ref)


def test_first_fetch_under_inference_mode(case):
    import torch
    ctx, slot = case
    with torch.inference_mode():
        first = slot()
    second = slot()
    same(first, want(ctx, slot))
    same(second, first)


def test_fetch_under_a_cuda_default_device(case):
    import torch
    ctx, slot = case
    torch.set_default_device("cuda:0")
    try:
        got = slot()
    finally:
        torch.set_default_device(None)
    same(got, want(ctx, slot))
