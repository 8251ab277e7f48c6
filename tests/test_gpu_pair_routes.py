"""The pair level tested pair by pair and by tensor-core tiles, on both sides of the count where one takes
over from the other, and the remaining rows extended in one launch: list, R_k and the candidates of
every level equal the oracle's pruned regain. The sketch is made with given numbers of hot estimators
per row, random bitmaps of several densities whose unions straddle the threshold."""
import numpy as np
import pytest

import oracle
from gpu_harness import assert_list_equal, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,n1,rest,log2_eta", [
    (1, 1, 1, 11), (7, 33, 40, 8), (512, 512, 24, 8), (513, 512, 24, 8), (300, 1100, 30, 9), (0, 5, 5, 8)])
@pytest.mark.parametrize("pair_level", [0, 1])
def test_pair_routes_match_oracle(n0, n1, rest, log2_eta, pair_level):
    q, r, k, eta = 11, 5, 60, 1 << log2_eta
    W = dict(params=dict(log2_eta=log2_eta, q=q, r=r, delta=7, k=k, theta=eta // 2), hash_seed=5)
    p, tabs, ctx = setup(W)
    ctx.tuning = dict(pair_level=pair_level)
    rng = np.random.default_rng(n0 * 10_000 + n1)
    sk = np.full((r, 1 << q, eta), 65535, dtype=np.uint16)
    for row, n in enumerate([n0, n1, rest, rest, rest]):
        for col in rng.choice(1 << q, n, replace=False):
            inside = rng.random(eta) < rng.choice([0.45, 0.6, 0.75, 0.95])
            sk[row, col, inside] = rng.integers(0, k, int(inside.sum()), dtype=np.uint16)
            sk[row, col, ~inside] = 60000
    glob = ctx.sketch()
    glob.load(sk.reshape(-1), 100)
    want = oracle.regain(p, tabs, sk.reshape(-1), "pruned")
    got = ctx.regain(glob, cap=1 << 17)
    assert_list_equal(got, want, f"{n0} x {n1}")
    assert ctx.stats()["level"] == [int(x) for x in want["levels"]]
    ctx.close()
