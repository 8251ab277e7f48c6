"""The rows after the pairs, extended from queues in one launch: long buckets, buckets cut into parts, queues that
fill and drain, every number of rows, and bitmaps of every form. List, R_k and candidates per level are the
oracle's pruned regain's. Candidate buffers that are too small, exactly as large as a level needs and
large enough are told apart, by the pairs tested one by one and by the later rows alike. And the time of few
candidates with long buckets is of the order of that of many candidates with short ones (the
same tests; extended depth first per lane, the first took 40 times the second's)."""
import numpy as np
import pytest

import oracle
import paper_1803_11036_gb300 as ssd
from gpu_harness import assert_list_equal, setup

pytestmark = pytest.mark.gpu
K = 60


def sketch(W, rows, dense, seed, columns=None):
    """Recorders with rows[i] columns of row i (or the given ones) inside the window with a probability of `dense`."""
    p = W["params"]
    eta, q, r = 1 << p["log2_eta"], p["q"], p["r"]
    rng = np.random.default_rng(seed)
    sk = np.full((r, 1 << q, eta), 65535, dtype=np.uint16)
    for row in range(r):
        cols = columns[row] if columns else rng.choice(1 << q, rows[row], replace=False)
        for col in cols:
            inside = rng.random(eta) < rng.choice(dense)
            sk[row, col, inside] = rng.integers(0, K, int(inside.sum()), dtype=np.uint16)
            sk[row, col, ~inside] = 60000
    return sk.reshape(-1)


def workload(log2_eta, q, r, delta, theta):
    return dict(params=dict(log2_eta=log2_eta, q=q, r=r, delta=delta, k=K, theta=theta), hash_seed=5)


@pytest.mark.parametrize("log2_eta,q,r,delta,rows,dense", [
    (8, 10, 5, 8, [3, 3, 200, 300, 60], [0.95]),               # long buckets (4 of them), cut into parts
    (8, 10, 5, 8, [40, 40, 12, 12, 12], [0.6, 0.95]),
    (9, 12, 4, 10, [20, 20, 40, 40], [0.7, 0.9]),
    (6, 10, 6, 6, [12, 12, 60, 60, 60, 20], [0.85, 0.97]),     # bitmaps of 2 words: hits one after another
    (7, 10, 8, 4, [9, 9, 120, 120, 120, 120, 120, 40], [0.97]),
    (5, 17, 3, 15, [30, 30, 300], [0.8, 0.9]),                 # the first of these rows is the last
    (5, 9, 7, 5, [6, 6, 30, 30, 30, 30, 8], [0.97])])
def test_rows_match_oracle(log2_eta, q, r, delta, rows, dense):
    W = workload(log2_eta, q, r, delta, (1 << log2_eta) // 2)
    p, tabs, ctx = setup(W)
    sk = sketch(W, rows, dense, r * 100 + log2_eta)
    glob = ctx.sketch()
    glob.load(sk, 100)
    want = oracle.regain(p, tabs, sk, "pruned")
    assert_list_equal(ctx.regain(glob, cap=1 << 18), want)
    assert ctx.stats()["level"] == [int(x) for x in want["levels"]]
    ctx.close()


def one_bucket(q, delta, counts):
    """Columns whose low q - delta bits are all 5 in the rows from 2 on: one long bucket per row."""
    rng = np.random.default_rng(1)
    cols = [rng.choice(1 << q, n, replace=False) for n in counts[:2]]
    return cols + [(np.arange(n) << (q - delta)) + 5 for n in counts[2:]]


def test_one_bucket_holds_every_column():
    W = workload(8, 12, 5, 7, 128)
    p, tabs, ctx = setup(W)
    sk = sketch(W, None, [0.9], 3, one_bucket(12, 7, [60, 60, 100, 100, 20]))
    glob = ctx.sketch()
    glob.load(sk, 100)
    want = oracle.regain(p, tabs, sk, "pruned")
    assert max(int(x) for x in want["levels"][2:]) > 1000
    assert_list_equal(ctx.regain(glob, cap=1 << 18), want)
    assert ctx.stats()["level"] == [int(x) for x in want["levels"]]
    ctx.close()


@pytest.mark.parametrize("level", [1, 2])
@pytest.mark.parametrize("short", [0, 1])
@pytest.mark.parametrize("call", ["regain", "close", "slot"])
def test_candidate_capacity(level, short, call):
    """A buffer that a level fills exactly is enough, one tuple less is SSD_ECAPACITY with the status bit."""
    import torch
    # the pairs are the largest level (1), or row 2 multiplies them (2)
    rows = [30, 30, 3, 3, 3] if level == 1 else [8, 8, 64, 1, 1]
    W = workload(8, 8 + 2, 5, 8, 128)
    p, tabs, ctx = setup(W)
    sk = sketch(W, rows, [0.9, 0.95], 7)
    want = oracle.regain(p, tabs, sk, "pruned")
    levels = [int(x) for x in want["levels"]]
    assert levels[level] == max(levels) and sorted(levels)[-2] < levels[level] - 1
    ctx.close()
    p, tabs, ctx = setup(W, ctb_capacity=levels[level] - short)
    glob = ctx.sketch()
    glob.load(sk, 100)
    none = torch.zeros((0, 2), dtype=torch.int32, device="cuda:0")
    run = {"regain": lambda: ctx.regain(glob, cap=1 << 16), "close": lambda: ctx.close_slot([glob]),
           "slot": lambda: ctx.slot([glob], [none])}[call]
    if short:
        with pytest.raises(ssd.SSDError) as err:
            run()
        assert err.value.code == ssd.SSD_ECAPACITY
        assert ctx.stats()["status"] & ssd.SSD_STATUS_CTB_OVERFLOW
    else:
        assert_list_equal(run(), want)
        assert ctx.stats()["status"] == 0 and ctx.stats()["level"] == levels
    ctx.close()


def test_time_does_not_depend_on_the_shape():
    import torch
    q, delta, le = 14, 6, 11
    W = workload(le, q, 5, delta, 2457)

    def tail_us(counts):
        p, tabs, ctx = setup(W)
        g = torch.Generator(device="cuda:0").manual_seed(1)
        rng = np.random.default_rng(1)
        sk = torch.full((5, 1 << q, 1 << le), -1, dtype=torch.int16, device="cuda:0")
        for row, n in enumerate(counts):   # (the last row's columns are hot, their unions not)
            cols = torch.from_numpy(rng.choice(1 << q, n, replace=False)).cuda()
            inside = torch.rand((n, 1 << le), generator=g, device="cuda:0") < (0.97 if row < 4 else 0.74)
            sk[row, cols] = torch.where(inside, 1, 30000).to(torch.int16)
        glob = ctx.sketch()
        glob.load_device(sk.reshape(-1), 40000)
        times = []
        for _ in range(7):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
            for e in ev:
                e.record()
            ctx.set_trace(*ev)
            ctx.regain(glob)
            ctx.set_trace()
            times.append(ev[1].elapsed_time(ev[2]) * 1e3)
        levels = ctx.stats()["level"]
        ctx.close()
        return sorted(times)[3], levels

    few, levels_few = tail_us([3, 3, 1 << q, 1 << q, 1024])      # 64 entries a bucket
    many, levels_many = tail_us([192, 192, 256, 256, 1024])      # 1 entry a bucket
    assert levels_few[3] > 30_000 and levels_many[3] > 30_000
    assert few < 6 * many, (few, many)
