"""Timed cases of the detector: whole slots, their parts and the served form, through the public
entry points of ``paper_1803_11036_gb300``.

A state holds what a monitor keeps between slots: one context, its sketches with a filled window, and
the pair buffers of several successive slots. Each pass takes the next slot's pairs, so a pass never
sees the pairs of the pass before, and the window stays in the steady state that the buffers,
cycled, keep up. Traffic follows the workload recipes of the repository (Zipf distinct-peer counts,
repeated pairs, planted super points, hot sources, lognormal packet counts per edge router), drawn
on the device from the seed alone and interleaved.
"""
import math

import numpy as np
import torch

import paper_1803_11036_gb300 as ssd
from paper_1803_11036_gb300.serve import Server, Slice

DEV = "cuda:0"


def _case(name, kind, packets, q, routers=1, log2_eta=11, r=5, delta=5, k=60, theta=1024, slots=8, counts="equal",
          rho=0.3, planted=20, lo=1500, hi=50_000, hot=0, sync=False, merged=False, cap=8192):
    """packets: per slot, all routers together; slots: distinct pair buffers of a state; planted hosts
    have lo..hi distinct peers per window; hot: sources that send 5 % of the packets each."""
    return dict(name=name, kind=kind, packets=packets, q=q, routers=routers, log2_eta=log2_eta, r=r, delta=delta, k=k,
                theta=theta, slots=slots, counts=counts, rho=rho, planted=planted, lo=lo, hi=hi, hot=hot, sync=sync,
                merged=merged, cap=cap)


def listed():
    return [
        # the smallest slots: a campus link's few hundred pairs, where launches and latency count
        _case("slot_tiny", "slot", 160, 9, log2_eta=6, delta=8, k=3, theta=40, planted=4, lo=45, hi=70, slots=3, sync=True),
        # the paper's own dimensions (Sec. 5), one router, the README's loop: the list on the host each slot
        _case("slot_paper", "slot", 1 << 18, 14, delta=6, k=4, lo=2000, hi=8000, slots=4, sync=True),
        # one core-link router at 40 Gb/s, lists left on the device (the pipelined form)
        _case("slot_corelink", "slot", 6_250_000, 18, planted=200),
        # 16 edge routers with lognormal packet counts, merged and regained centrally
        _case("slot_edges", "slot", 11_673_000, 16, routers=16, delta=6, planted=200, slots=4, counts="lognormal"),
        # 32 routers at 100 Gb/s: hosts straddling the threshold, repeated pairs and ten hot sources
        _case("slot_stress", "slot", 15_600_000, 16, routers=32, delta=6, k=300, rho=0.6, planted=5000, lo=900, hi=1150,
              hot=10, slots=4),
        # many resident routers served from pinned host memory, all slices ready at once
        _case("served", "served", 8_040_008, 17, routers=8, counts="uniform", slots=2, cap=4096),
        # Algorithm 2 alone on a core link: a monitor that scans in several batches per slot
        _case("scan_corelink", "scan", 6_250_000, 18, planted=200, slots=4),
        # bidirectional detection with two host groups per side: four views of the same pairs, one launch
        _case("scan_views", "views", 1_562_501, 16, delta=6, planted=50, slots=4),
        # scan_batch then close_slot keeping the merged sketch, a few small edge routers
        _case("batch_close", "batch", 520_003, 14, routers=4, delta=6, k=6, planted=30, hi=12_000, slots=6,
              counts="lognormal", merged=True, sync=True),
        # the plain method of the paper, one call per step: advance, scan per router, merge, regain
        _case("plain_steps", "plain", 2_000_000, 16, routers=4, delta=6, planted=50, slots=6, counts="uniform",
              merged=True, sync=True),
        # regaining a wide merged sketch: thousands of hosts about the threshold
        _case("regain_wide", "regain", 4_000_000, 16, delta=6, k=300, rho=0.6, planted=3000, lo=900, hi=1150, slots=4,
              sync=True),
        # checkpoint, and the fold of two routers' exported recorders (routers spread over machines), and resume
        _case("checkpoint", "checkpoint", 1_000_000, 16, routers=2, delta=6, slots=2),
    ]


def draw(rng):
    kind = rng.choice(["slot", "slot", "slot", "served", "scan", "views", "batch", "plain", "regain", "checkpoint"])
    r = rng.choice([4, 5, 5, 5, 6])
    log2_eta = rng.choice([6, 8, 9, 10, 11, 11, 11, 12])
    routers = 1
    if kind in ("slot", "batch", "plain"):
        routers = rng.choice([1, 1, 2, 3, 5, 8, 13, 16, 24])
    if kind == "served":
        routers = rng.choice([2, 3, 6])
    if kind == "checkpoint":
        routers = 2
    k = rng.choice([1, 4, 6, 17, 60, 300]) if kind != "regain" else rng.choice([6, 17, 60, 300])
    slots = min(4, max(2, k)) if k > 1 else 2
    packets = int(math.exp(rng.uniform(math.log(200), math.log(4_000_000)))) | rng.randint(0, 1)
    # columns for about a tenth of the estimator's recorders per window, as the repository's workloads have
    q = min(18, max(12, math.ceil(math.log2(slots * packets / (0.1 * (1 << log2_eta)) + 1))))
    while q > 12 and routers * r * 2 ** (q + log2_eta + 1) > 6 << 30:
        q -= 1
    packets = min(packets, int(0.2 * (1 << log2_eta) * (1 << q) / slots))
    theta = max(24, (1 << log2_eta) // 2 + rng.randint(-7, 7))
    return dict(kind=kind, packets=packets, q=q, routers=routers, log2_eta=log2_eta, r=r,
                delta=-(-(32 - q) // (r - 2)), k=k, theta=theta, slots=slots,
                counts=rng.choice(["equal", "uniform", "lognormal"]), rho=rng.choice([0.0, 0.3, 0.6]),
                planted=min(rng.choice([2, 10, 40]), packets // 200 + 1), lo=theta, hi=4 * theta,
                hot=rng.choice([0, 0, 3]), sync=kind in ("plain", "regain") or rng.random() < 0.4,
                merged=rng.random() < 0.4 or kind == "plain", cap=4096)


def _fmix(h):
    """A 32-bit mix of int64 tensors holding unsigned 32-bit values."""
    h = h & 0xFFFFFFFF
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & 0xFFFFFFFF
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & 0xFFFFFFFF
    return h ^ (h >> 16)


class _Traffic:
    def __init__(self, c, seed):
        self.c = c
        self.g = torch.Generator(device=DEV).manual_seed(seed)
        self.key = (seed * 2654435761) & 0xFFFFFFFF
        rng = np.random.RandomState(seed & 0x7FFFFFFF)
        # distinct pairs of a window: a tenth of the recorders of a row, sources of Zipf(1.1) degree
        eta, cols = 1 << c["log2_eta"], 1 << c["q"]
        cap = max(2, min(512, c["theta"] // 2))
        w = np.arange(1, cap + 1, dtype=np.float64) ** -1.1
        mean = float((np.arange(1, cap + 1) * w).sum() / w.sum())
        # (of all routers together: router j's sources start at 0.7 * j * n_src)
        pairs = min(0.1 * eta * cols, 4.0 * c["slots"] * c["packets"])
        n_src = max(8, int(pairs / mean / (1 + 0.7 * (c["routers"] - 1 if c["kind"] != "served" else 0))))
        cdf = torch.from_numpy(np.cumsum(w) / w.sum()).to(DEV)
        u = torch.rand(n_src, generator=self.g, device=DEV, dtype=torch.float64)
        self.cum = torch.cumsum(torch.searchsorted(cdf, u).clamp_(max=cap - 1) + 1, 0)
        self.total = int(self.cum[-1])
        self.peers = torch.from_numpy(rng.randint(c["lo"], c["hi"] + 1, max(1, c["planted"])).astype(np.int64)).to(DEV)
        self.n_src, self.rng = n_src, rng

    def counts(self):
        """Packets of each router in one slot, about c["packets"] in all."""
        c, n = self.c, self.c["routers"]
        if c["counts"] == "lognormal":
            w = self.rng.lognormal(0.0, 1.0, n)
        elif c["counts"] == "uniform":
            w = self.rng.uniform(0.01, 2.0, n)
        else:
            w = np.ones(n)
        return [max(1, int(c["packets"] * x / w.sum())) for x in w]

    def _rand(self, n):
        return torch.rand(n, generator=self.g, device=DEV, dtype=torch.float64)

    def slot(self, t, j, n):
        """The pairs of router j in slot t: an int32 tensor (n, 2)."""
        c = self.c
        m = -(-self.peers // c["slots"])
        host = torch.repeat_interleave(torch.arange(len(m), device=DEV), m)
        at = torch.arange(len(host), device=DEV) - (torch.cumsum(m, 0) - m)[host]
        idx = (t * m[host] + at) % self.peers[host]
        if c["routers"] > 1:   # a planted host's peer always enters through the same router
            keep = _fmix(host * 7919 + idx) % c["routers"] == j
            host, idx = host[keep], idx[keep]
        host, idx = host[: n // 2], idx[: n // 2]
        src, peer = [host + 0x40000000], [idx]
        for h in range(c["hot"]):
            cnt = n // 20
            src.append(torch.full((cnt,), 0x50000000 + h, device=DEV))
            peer.append((self._rand(cnt) * 256).long())
        left = n - sum(len(x) for x in src)
        pair = (self._rand(left) * self.total).long().clamp_(max=self.total - 1)
        s = torch.searchsorted(self.cum, pair, right=True)
        p = pair - torch.where(s > 0, self.cum[(s - 1).clamp_(min=0)], 0)
        if left and c["rho"] > 0:   # repeats of earlier pairs of the slot
            back = (self._rand(left) * torch.arange(left, device=DEV)).long()
            again = self._rand(left) < c["rho"]
            s, p = torch.where(again, s[back], s), torch.where(again, p[back], p)
        # routers see overlapping source sets: 70 % of a router's sources are its own
        src.append(s + (j * int(0.7 * self.n_src)))
        peer.append(p)
        s, p = torch.cat(src), torch.cat(peer)
        order = torch.randperm(n, generator=self.g, device=DEV)
        s, p = s[order], p[order]
        cip = _fmix(s ^ self.key)
        oip = _fmix(_fmix(p ^ cip) + s)
        return torch.stack((cip, oip), 1).to(torch.int32).contiguous()


def _tables(seed):
    return np.random.RandomState((seed ^ 0x5EED) & 0x7FFFFFFF).randint(0, 1 << 32, 2048, dtype=np.uint64).astype(np.uint32)


def _outputs(cap):
    return (torch.zeros(cap, dtype=torch.int32, device=DEV), torch.zeros(cap, dtype=torch.int32, device=DEV),
            torch.zeros(1, dtype=torch.int64, device=DEV))


def prepare(case, seed):
    c = case
    params = ssd.make_params({f: c[f] for f in ("log2_eta", "q", "r", "delta", "k", "theta")})
    traffic, tables, n = _Traffic(c, seed), _tables(seed), c["routers"]
    if c["kind"] == "served":
        server = Server(params, tables, max_inflight=8, list_cap=c["cap"], max_slice_pairs=2 * c["packets"] + 64)
        slots = [[traffic.slot(t, j, m).cpu().pin_memory() for j, m in enumerate(traffic.counts())] for t in range(c["slots"])]
        st = dict(case=c, server=server, slots=slots, at=0)
        run(st)   # the routers are resident and the window has a slot
        st["views"] = _views([server.tenants[j].sketch for j in range(n)])
        return st
    ctx = ssd.Context(params, tables)
    st = dict(case=c, ctx=ctx, at=0)
    if c["kind"] == "views":
        st["routers"] = [ctx.sketch().set_view(side, 1, group) for side in (0, 1) for group in (0, 1)]
    else:
        st["routers"] = [ctx.sketch() for _ in range(n)]
    st["merged"] = ctx.sketch() if c["merged"] or c["kind"] in ("regain", "plain", "checkpoint") else None
    st["slots"] = [[traffic.slot(t, j, m) for j, m in enumerate(traffic.counts())] for t in range(c["slots"])]
    st["out"] = _outputs(c["cap"])
    if c["kind"] != "regain":
        ctx.reserve(max(sum(len(p) for p in s) for s in st["slots"]))
    # a filled window: every buffer has been a slot once
    for pairs in st["slots"]:
        if c["kind"] == "views":
            ctx.scan_batch(st["routers"], pairs * 4)
        else:
            ctx.scan_batch(st["routers"], pairs)
        ctx.advance(st["routers"])
    if c["kind"] == "regain":
        ctx.merge(st["routers"], st["merged"])
    st["views"] = _views(st["routers"] + [st["merged"]])
    if c["kind"] == "checkpoint":
        count = ctx.sketch_bytes // 2
        st["images"] = [torch.empty(count, dtype=torch.int16, device=DEV) for _ in range(n)]
    return st


def _views(sketches):
    """The stored recorders of the sketches, sharing their memory: each view keeps its sketch alive."""
    views = []
    for sketch in sketches:
        if sketch is not None:
            views.append(sketch.device_view())
            views[-1].sketch = sketch
    return views


def _list(c, ips, rk):
    """A list of hosts and their R_k as one array of its capacity."""
    out = np.zeros((2, c["cap"]), dtype=np.uint32)
    out[0, : len(ips)] = ips
    out[1, : len(rk)] = rk
    return out


def run(state):
    c, at = state["case"], state["at"]
    pairs = state["slots"][at % len(state["slots"])]
    state["at"] = at + 1
    kind = c["kind"]
    if kind == "served":
        server = state["server"]
        server.results = []
        res = server.run([Slice(j, p, 0.0) for j, p in enumerate(pairs)], realtime=False)
        lists = [_list(c, r.ips, r.rk) for r in sorted(res, key=lambda r: (r.router, r.slot))]
        return lists, state.get("views")
    ctx, routers, merged = state["ctx"], state["routers"], state["merged"]
    if kind == "slot":
        ctx.slot(routers, pairs, merged, out=state["out"], sync=c["sync"])   # with sync also as host arrays
        return state["out"], state["views"]
    if kind == "batch":
        ctx.scan_batch(routers, pairs)
        ctx.close_slot(routers, merged, out=state["out"], sync=c["sync"])
        return state["out"], state["views"]
    if kind == "scan":
        ctx.scan(routers[0], pairs[0])
        return state["views"]
    if kind == "views":
        ctx.scan_batch(routers, pairs * 4)
        return state["views"]
    if kind == "plain":
        ctx.advance(routers)
        for router, p in zip(routers, pairs):
            ctx.scan(router, p)
        ctx.merge(routers, merged)
        return _list(c, *ctx.regain(merged, cap=c["cap"])), state["views"]
    if kind == "regain":
        return _list(c, *ctx.regain(merged, cap=c["cap"])), state["views"][-1:]
    # checkpoint: each router's recorders out, their fold, and the fold resumed as the merged sketch
    images = state["images"]
    for router, image in zip(routers, images):
        router.export_device(image)
    ctx.min_merge(images[0], images)
    merged.load_device(images[0], routers[0].slot)
    return images, state["views"][-1:]


def work(case):
    """Every sketch that the path has to look through is read once, the pairs are read once, each touched
    recorder is written (two bytes per pair and row), and a merged sketch is written whole. A scan alone
    reads no recorder."""
    c = case
    sketch = c["r"] * 2 ** (c["q"] + c["log2_eta"] + 1)
    touched = c["packets"] * (8 + 2 * c["r"])
    n = c["routers"]
    kind = c["kind"]
    if kind in ("slot", "batch", "served"):
        moved = n * sketch + touched + (sketch if c["merged"] else 0)
    elif kind == "scan":
        moved = touched
    elif kind == "views":
        moved = c["packets"] * (8 + 4 * c["r"])
    elif kind == "plain":   # advance and merge read the routers once each, regain reads the merged sketch
        moved = 2 * n * sketch + touched + 2 * sketch
    elif kind == "regain":
        moved = sketch
    else:   # two exports, the fold of two into one, one import
        moved = 2 * n * sketch + (n + 1) * sketch + 2 * sketch
    return {"bytes": moved, "flops": 0}
