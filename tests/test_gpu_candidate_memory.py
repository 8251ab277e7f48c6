"""A context holds the second candidate buffer only where a launch per row reads and writes it: without pruning, or
without the bucket index."""
import pytest

import paper_1803_11036_gb300 as ssd
import trafficgen as tg

pytestmark = pytest.mark.gpu
CAP = 1 << 26   # tuples of r = 5 words: 1.25 GiB a buffer


@pytest.mark.parametrize("q,delta,flags,buffers", [(14, 6, 0, 1), (14, 6, ssd.SSD_NO_PRUNE, 2), (21, 4, 0, 2)])
def test_candidate_buffers(q, delta, flags, buffers):
    import torch
    params = ssd.make_params(dict(log2_eta=5, q=q, r=5, delta=delta, k=4, theta=16), flags, ctb_capacity=CAP)
    small = ssd.make_params(dict(log2_eta=5, q=q, r=5, delta=delta, k=4, theta=16), flags, ctb_capacity=1 << 10)

    def held(prm):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = ssd.Context(prm, tg.hash_tables(1))
        after = torch.cuda.mem_get_info()[0]
        ctx.close()
        return before - after

    held(small)
    one = CAP * 5 * 4
    assert abs(held(params) - held(small) - buffers * one) < one // 8
