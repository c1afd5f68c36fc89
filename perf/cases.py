"""The work that users of this library have it do, as measurable cases.

Each case is a program a user writes against ``paper_2211_15963_gb300.dbnet``:
a network stepped and read, an HMDA cycle, a batch of served requests, an
allocation-free run.  ``prepare`` makes what such a program has in hand (the
host graph, or the network, ensemble or server that it keeps), ``run`` is one
pass of its loop.  Graphs are drawn on the GPU from the seed with the shapes
of the paper's networks: 4:1 excitatory to inhibitory neurons per region, most
edges within the region at short delays, the rest from excitatory neurons to
other regions at long ones, lognormal weights.

Spiking networks are chaotic: 32-bit and 64-bit trajectories part within tens
of milliseconds, so ``exact`` gives values only where a pass starts from the
initial state and is short (closed loop, allocation-free run), and the
others' state, spikes and counts are compared with another run's alone.
"""
import math
import types

import numpy as np
import torch

from paper_2211_15963_gb300 import dbnet

# Constant currents for about 10 Hz at an in-degree of 100, 300 and 1,000 (the
# serving workload's table); conductances scale with 100 / in-degree.
DRIVE = ((100, 0.75084), (300, 2.36363), (1000, 4.88653))


# ------------------------------------------------------------------ cases ----
def listed():
    return [
        # A closed loop on the small network: advance 1 ms, look at the state,
        # decide, go on.  All latency.
        dict(name="closed_loop_10k", kind="loop", neurons=10_000, regions=1, k=100, steps=10),
        # A quick look at a small ragged network: build it, run 100 ms, take
        # the spikes, the state and the BOLD, drop it.
        dict(name="one_shot_12k", kind="oneshot", neurons=12_345, regions=3, k=100, steps=1000),
        # The small network of the parity tests simulated for a second.
        dict(name="small_10k_1s", kind="net", neurons=10_000, regions=1, k=100, steps=10_000),
        # A run inside a caller that may not allocate: graph and state are the
        # caller's device arrays.
        dict(name="noalloc_30k", kind="noalloc", neurons=30_011, regions=5, k=150, steps=200),
        # The task variant on odd, ragged regions: Ornstein-Uhlenbeck
        # background and Gamma-distributed injected currents.
        dict(name="task_150k", kind="net", neurons=149_993, regions=7, k=300, steps=1000, ragged=True,
             ou=True),
        # Two float32 weights per edge (one per channel) on ragged regions.
        dict(name="two_weights_300k", kind="net", neurons=300_007, regions=23, k=400, steps=1000,
             ragged=True, two_weights=True),
        # The mid-size network of the benchmark at 15 Hz, 100 ms a pass.
        dict(name="mid_2m", kind="net", neurons=2_000_000, regions=100, k=1000, steps=1000, drive=7.22,
             hz=15.0),
        # Five million neurons in regions of 100,000 like the largest
        # network's: the accumulators no longer share the L2 with the rest.
        dict(name="large_5m", kind="net", neurons=5_000_000, regions=50, k=400, steps=500),
        # The NEST-comparison shape: 1 ms steps, in-degree 100, no delay
        # beyond one step; the state's traffic dominates.
        dict(name="nest_4m_1ms", kind="net", neurons=4_000_000, regions=200, k=100, steps=500, nest=True,
             hz=12.0),
        # Cortical columns: heavy-tailed out-degrees, spikes handed on at the
        # edges of 1 ms bins.
        dict(name="columns_500k", kind="net", neurons=500_000, regions=25, k=500, steps=1000, columns=True),
        # One HMDA cycle of the 64-member ensemble: 100 ms of every member,
        # then the diffusion analysis against an observed BOLD sample.
        dict(name="hmda_64x100k", kind="hmda", neurons=100_000, regions=20, k=500, members=64, steps=1000),
        # Eight requests of mixed sizes served together, each uploading its
        # own graph.
        dict(name="serve_8", kind="serve", neurons=120_000, regions=12, k=300, requests=8, steps=2000),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["loop", "oneshot", "net", "net", "net", "net", "noalloc", "hmda", "serve"])
    if kind == "loop":
        return dict(kind=kind, neurons=size(2_000, 60_000), regions=rng.randint(1, 6), k=size(60, 300),
                    steps=rng.choice([1, 5, 10, 20]))
    if kind == "oneshot":
        return dict(kind=kind, neurons=size(2_000, 80_000), regions=rng.randint(1, 8), k=size(60, 300),
                    steps=rng.randint(200, 1500))
    if kind == "noalloc":
        return dict(kind=kind, neurons=size(1_500, 60_000), regions=rng.randint(1, 12), k=size(50, 200),
                    steps=rng.randint(50, 300))
    if kind == "hmda":
        return dict(kind=kind, neurons=size(10_000, 60_000), regions=rng.randint(2, 30), k=size(100, 400),
                    members=rng.randint(8, 64), steps=10 * rng.randint(20, 80), observer=rng.choice(["diffusion", "global"]))
    if kind == "serve":
        return dict(kind=kind, neurons=size(20_000, 150_000), regions=rng.randint(2, 20), k=size(100, 300),
                    requests=rng.randint(2, 8), steps=rng.randint(500, 2000))
    n = size(10_000, 3_000_000)
    k = min(size(100, 1000), max(100, int(4e8 // n)))
    c = dict(kind="net", neurons=n, regions=max(1, min(rng.randint(1, 120), n // 3_000)), k=k,
             steps=rng.randint(300, 1200))
    form = rng.choice(["plain", "plain", "ragged", "ou", "two_weights", "columns", "nest"])
    if form in ("ragged", "ou", "two_weights"):
        c["ragged"] = True
    if form != "plain" and form != "ragged":
        c[form] = True
    if form == "nest":
        c["k"] = min(k, 150)
    return c


# ----------------------------------------------------------------- graphs ----
def sizes_of(case):
    """Region sizes: equal, or ragged by a fixed rule of the case's numbers."""
    n, r = case["neurons"], case["regions"]
    if not case.get("ragged") and n % r == 0:
        return [n // r] * r
    share = np.random.RandomState(n % 65_521).uniform(0.4, 1.6, r)
    s = np.maximum((share / share.sum() * n).astype(np.int64), 8)
    s[-1] += n - s.sum()
    return [int(x) for x in s]


def drive_of(k):
    if k <= DRIVE[0][0]:
        return DRIVE[0][1]
    for (k0, v0), (k1, v1) in zip(DRIVE, DRIVE[1:]):
        if k <= k1:
            return v0 * (v1 / v0) ** (math.log(k / k0) / math.log(k1 / k0))
    return DRIVE[-1][1]


def region_params(case):
    k = case["k"]
    g = [0.006, 0.00002, 0.6, 0.002]
    p = dict(C=0.5, gL=0.025, VL=-70.0, Vth=-50.0, Vreset=-55.0, Tref=2.0, Vu=(0.0, 0.0, -70.0, -100.0),
             tau_u=(2.0, 100.0, 10.0, 100.0), drive_rate_hz=10.0, drive_K=1.0, w_ext=2.0)
    if case.get("nest"):
        p.update(I_ext=0.9, g_u=tuple(0.2 * x * 100 / k for x in g))
    else:
        p.update(I_ext=case.get("drive") or drive_of(k), g_u=tuple(x * 100 / k for x in g))
    if case.get("ou"):
        p.update(ou_mu=0.1, ou_sigma=0.2, ou_tau=10.0, iext_shape=25.0)
    return p


def delay_ranges(case):
    if case.get("nest"):
        return (1, 1), (1, 1)
    if case.get("columns"):
        return (1, 20), (20, 100)
    if case["kind"] == "noalloc":
        return (1, 15), (15, 30)
    if case["regions"] == 1:
        return (1, 20), (1, 20)
    return (1, 50), (50, 200)


class Drawn:
    """Edges drawn block by block on the GPU and kept in host memory (pinned,
    as a program that loads a network does), or on the GPU."""

    def __init__(self, n_edges, host, float_weights, two):
        def room(dtype):
            return torch.empty(n_edges, dtype=dtype, pin_memory=True) if host else \
                torch.empty(n_edges, dtype=dtype, device="cuda")
        wt = torch.float32 if float_weights else torch.int16
        self.col, self.delay, self.w = room(torch.int32), room(torch.uint8), room(wt)
        self.w2 = room(wt) if two else None
        self.float_weights, self.at = float_weights, 0

    def add(self, gen, col, delay):
        n = col.numel()
        s = slice(self.at, self.at + n)
        self.col[s].copy_(col.reshape(-1), non_blocking=True)
        self.delay[s].copy_(delay.reshape(-1), non_blocking=True)
        for to in (self.w, self.w2):
            if to is not None:
                w = torch.randn(n, generator=gen, device="cuda").mul_(0.5).sub_(1.0).exp_()
                to[s].copy_(w if self.float_weights else w.bfloat16().view(torch.int16), non_blocking=True)
        self.at += n


def sorted_uniforms(gen, rows, k):
    """k ascending uniforms per row: partial sums of exponentials over their total."""
    e = torch.empty(rows, k + 1, device="cuda").exponential_(generator=gen)
    s = torch.cumsum(e, 1)
    return s[:, :k] / s[:, k:]


def sorted_delays(gen, rows, k, lo, hi):
    if lo == hi:
        return torch.full((rows, k), lo, dtype=torch.uint8, device="cuda")
    u = sorted_uniforms(gen, rows, k)
    return u.mul_(hi - lo + 1).to(torch.int32).clamp_(max=hi - lo).add_(lo).to(torch.uint8)


def make_graph(case, seed, host=True):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    sizes, k = sizes_of(case), case["k"]
    R, N = len(sizes), sum(sizes)
    ro = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n_exc = np.array([int(round(0.8 * s)) for s in sizes], np.int32)
    within, cross = delay_ranges(case)
    start = torch.tensor(ro[:-1].astype(np.int64), device="cuda")
    size = torch.tensor(sizes, device="cuda")
    # cross-region strengths: a sparse lognormal row per source region
    cdf = None
    if R > 1:
        m = torch.randn(R, R, generator=gen, device="cuda").exp_()
        m *= torch.rand(R, R, generator=gen, device="cuda") < max(0.3, 1.5 / (R - 1))
        m += 1e-6
        m.fill_diagonal_(0.0)
        cdf = torch.cumsum(m / m.sum(1, keepdim=True), 1)

    def cross_targets(r, shape):
        t = torch.bucketize(torch.rand(shape, generator=gen, device="cuda"), cdf[r]).clamp_(max=R - 1)
        t = torch.where(t == r, (t + 1) % R, t)
        u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
        return (start[t] + (u * size[t]).long()).to(torch.int32)

    def within_targets(r, shape):
        return torch.randint(int(ro[r]), int(ro[r + 1]), shape, generator=gen, device="cuda", dtype=torch.int32)

    two, fw = bool(case.get("two_weights")), bool(case.get("two_weights"))
    # of k edges per neuron 80 % stay in the region; the rest leave from its
    # excitatory neurons, a quarter more from each of those
    kw = k if R == 1 else int(round(0.8 * k))
    kc = 0 if R == 1 else int(round(1.25 * (k - kw)))
    deg = torch.empty(N, dtype=torch.int64, device="cuda")
    for r in range(R):
        a, e, b = int(ro[r]), int(ro[r] + n_exc[r]), int(ro[r + 1])
        deg[a:e], deg[e:b] = kw + kc, kw
    if case.get("columns"):  # heavy-tailed rows
        f = torch.randn(N, generator=gen, device="cuda").mul_(0.6).sub_(0.18).exp_()
        deg = (deg * f).long().clamp_(1, 8 * k)
    row_ptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=row_ptr[1:])
    out = Drawn(int(row_ptr[-1]), host, fw, two)
    for r in range(R):
        a, e, b = int(ro[r]), int(ro[r] + n_exc[r]), int(ro[r + 1])
        if case.get("columns"):
            row = torch.repeat_interleave(torch.arange(b - a, device="cuda"), deg[a:b])
            far = (torch.rand(row.numel(), generator=gen, device="cuda") < (kc / (kw + kc) if kc else 0.0)) & (row < e - a)
            u = torch.rand(row.numel(), generator=gen, device="cuda")
            lo = torch.where(far, cross[0], within[0])
            d = lo + (u * torch.where(far, cross[1] - cross[0] + 1, within[1] - within[0] + 1)).long()
            key = torch.sort(row * 512 + d * 2 + far)[0]
            far, d = (key & 1).bool(), ((key >> 1) & 255).to(torch.uint8)
            col = within_targets(r, key.shape)
            if R > 1:
                col = torch.where(far, cross_targets(r, key.shape), col)
            out.add(gen, col, d)
            continue
        for rows, far in ((e - a, kc), (b - e, 0)):
            for at in range(0, rows, max(1, (1 << 25) // (kw + kc))):
                n = min(rows - at, max(1, (1 << 25) // (kw + kc)))
                d = sorted_delays(gen, n, kw, *within)
                col = within_targets(r, (n, kw))
                if far:
                    d = torch.cat([d, sorted_delays(gen, n, far, *cross)], 1)
                    col = torch.cat([col, cross_targets(r, (n, far))], 1)
                out.add(gen, col, d)
    torch.cuda.current_stream().synchronize()
    g = types.SimpleNamespace(n_neurons=N, n_regions=R, region_offsets=ro, n_exc=n_exc,
                              row_ptr=row_ptr.cpu().numpy() if host else row_ptr, col=out.col, delay=out.delay)
    if fw:
        g.weight, g.weight2 = out.w, out.w2
    else:
        g.w_bf16 = out.w
    return g


# ------------------------------------------------------------ preparation ----
def options(case, seed, **over):
    o = dict(seed=int(seed) % (1 << 31) + 1, tr_ms=20.0)
    if case.get("nest"):
        o.update(dt_ms=1.0, bin_ms=1.0)
    if case.get("columns"):
        o.update(bin_spikes=1)
    o.update(over)
    return o


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        g = make_graph(case, seed, host=False)
        n_pad = -(-g.n_neurons // 1024) * 1024
        cap = g.n_neurons * 8
        return dict(case=case, graph=g, params=region_params(case), options=options(case, seed),
                    V=torch.zeros(n_pad, device="cuda"), J=torch.zeros(4, n_pad, device="cuda"),
                    ref=torch.zeros(n_pad, dtype=torch.uint8, device="cuda"),
                    step=torch.zeros(cap, dtype=torch.int32, device="cuda"),
                    id=torch.zeros(cap, dtype=torch.int32, device="cuda"),
                    spikes=torch.zeros(cap, dtype=torch.int64, device="cuda"))
    if kind == "oneshot":
        return dict(case=case, graph=make_graph(case, seed), params=region_params(case),
                    options=options(case, seed, raster_capacity=case["neurons"] * 20))
    if kind == "loop":
        net = dbnet.Network(make_graph(case, seed), region_params(case), options(case, seed))
        return dict(case=case, net=net)
    if kind == "net":
        # a network past its onset, its launch shape chosen by the library
        net = dbnet.Network(make_graph(case, seed), region_params(case), options(case, seed, autotune_at=256))
        net.step(512)
        for _ in range(16):
            if net.stats()["autotuned"]:
                break
            net.step(512)
        net.sync()
        return dict(case=case, net=net)
    rng = np.random.default_rng(seed)
    if kind == "hmda":
        M, R = case["members"], case["regions"]
        theta = rng.uniform(-0.69, 0.69, (M, R, 2))
        enkf = dict(mode=dbnet.DBENS_GLOBAL if case.get("observer") == "global" else dbnet.DBENS_DIFFUSION)
        g = make_graph(case, seed)
        o = options(case, seed, tr_ms=case["steps"] * 0.1, autotune_at=256)
        ens = dbnet.Ensemble(g, region_params(case), M, theta, o, enkf)
        for _ in range(16):
            ens.step(case["steps"])
            if ens.member_stats(0)["autotuned"]:
                break
        # what the scanner shows: the forecast of one member, with noise
        y = ens.read()[2][0] * rng.uniform(0.9, 1.1, R)
        return dict(case=case, ens=ens, y=y, eps=rng.standard_normal((M, R)), xi=rng.standard_normal((M, R, 2)))
    if kind == "serve":
        mix, todo = np.random.RandomState(case["neurons"] % 65_521), []  # the mix is the case's, the networks the seed's
        for i in range(case["requests"]):
            n = max(2_000, int(case["neurons"] * mix.uniform(0.1, 1.0)))
            c = dict(case, neurons=n, regions=max(1, min(case["regions"], n // 2_000)), ragged=True,
                     k=max(60, int(case["k"] * mix.uniform(0.4, 1.0))))
            todo.append((make_graph(c, seed * 31 + i), region_params(c), int(case["steps"] * mix.uniform(0.3, 1.0))))
        srv = dbnet.Server(max_neurons=case["neurons"] * case["requests"] + 1024 * 64, max_requests=16,
                           max_regions=case["regions"] * 16, max_delay=200, arena_bytes=8 << 30,
                           run=options(case, seed))
        return dict(case=case, srv=srv, todo=todo, served=0, capacity=4 * case["neurons"])
    raise ValueError(kind)


def state_of(net):
    V, J, ref = net.state()
    return dict(V=V, J=J, ref=ref, bw=net.bw())


def raster(step, ids, room):
    """The spikes in a buffer of the room they may take, as a program that keeps one image a pass does."""
    out = np.full((2, room), -1, np.int32)
    out[0, :len(step)], out[1, :len(ids)] = step, ids
    return out


# ------------------------------------------------------------------ a pass ----
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("loop", "net"):
        s["net"].step(case["steps"])
        out = state_of(s["net"])
        if kind == "net":
            st = s["net"].stats()
            out.update(spikes=st["spikes"], events=st["events"])
        return out
    if kind == "oneshot":
        net = dbnet.Network(s["graph"], s["params"], s["options"])
        net.step(case["steps"])
        out = state_of(net)
        out.update(raster=raster(*net.spikes(), s["options"]["raster_capacity"]), bold=net.bold())
        net.close()
        return out
    if kind == "noalloc":
        g = s["graph"]
        n, events = dbnet.dbnet_run_noalloc(g.n_neurons, g.region_offsets, g.n_exc, g.row_ptr, g.col, g.w_bf16,
                                            g.delay, s["params"], s["options"], case["steps"], s["V"], s["J"],
                                            s["ref"], s["step"], s["id"])
        # spikes come unordered within a step: the caller orders them
        N = g.n_neurons
        s["spikes"].fill_(-1)
        s["spikes"][:n] = torch.sort(s["step"][:n].long() * N + s["id"][:n])[0]
        return dict(V=s["V"][:N], J=s["J"][:, :N], ref=s["ref"][:N], spikes=s["spikes"], events=events)
    if kind == "hmda":
        e = s["ens"]
        e.step(case["steps"])
        forecast = e.assimilate(s["y"], s["eps"], s["xi"])
        theta, bw, y = e.read()
        return dict(forecast=forecast, theta=theta, bw=bw, y=y)
    srv = s["srv"]
    s["served"] += 1
    ids = [srv.submit(g, p, n, seed=s["served"] * 97 + i, raster_capacity=s["capacity"])
           for i, (g, p, n) in enumerate(s["todo"])]
    srv.drain()
    out = []
    for i in ids:
        out.append(dict(bold=srv.bold(i), raster=raster(*srv.spikes(i), s["capacity"])))
        srv.release(i)
    return out


# -------------------------------------------------------------------- work ----
def work(case):
    """Bytes of one pass: per neuron and step the state read and written once
    (58; four accumulator channels 74; background current and factor 12 more),
    per synaptic event its record and its accumulator (14, or 24), and the
    results.  Flops: about 40 per neuron and step."""
    n, steps, kind = case["neurons"], case["steps"], case["kind"]
    dt = 1e-3 if case.get("nest") else 1e-4
    two = bool(case.get("two_weights"))
    copies = case.get("members", 1)
    if kind == "serve":  # sizes and lengths are drawn: 0.1 to 1 and 0.3 to 1 of the case's
        copies, steps = 0.55 * case["requests"], 0.65 * case["steps"]
    per = 58 + (16 if two else 0) + (12 if case.get("ou") else 0)
    events = n * case.get("hz", 10.0) * dt * case["k"]
    b = copies * steps * (n * per + events * (24 if two else 14))
    b += n * 25 if kind in ("loop", "net", "oneshot", "noalloc") else 0
    if kind in ("oneshot", "serve"):  # the graph comes in: 7 bytes an edge, 6 kept
        b += copies * n * case["k"] * 13
    return dict(bytes=float(b), flops=float(copies * steps * (40.0 * n + 2.0 * events)))


# --------------------------------------------------------- 64-bit reference ----
def mul64(a, b):
    """High and low words of the product of a constant and an array of uint64."""
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    a = np.uint64(a)
    al, ah, bl, bh = a & m, a >> s, b & m, b >> s
    ll, lh, hl = al * bl, al * bh, ah * bl
    mid = (ll >> s) + (lh & m) + (hl & m)
    return ah * bh + (lh >> s) + (hl >> s) + (mid >> s), a * b


def philox(c0, c1, c2, key):
    """Philox4x64-10 (Salmon et al., SC'11) at counters (c0, c1, c2, 0)."""
    c = [np.full_like(c1, c0), c1.copy(), np.full_like(c1, c2), np.zeros_like(c1)]
    k0, k1 = key
    for _ in range(10):
        h0, l0 = mul64(0xD2E7470EE14C6C93, c[0])
        h1, l1 = mul64(0xCA5A826395121157, c[2])
        c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
        k0 = (k0 + 0x9E3779B97F4A7C15) & (2**64 - 1)
        k1 = (k1 + 0xBB67AE8584CAA73B) & (2**64 - 1)
    return np.stack(c, 1).reshape(-1)


def simulate64(case, seed, g):
    """The network from its initial state, in 64 bits: state and spikes."""
    def host(a):
        return a.cpu().numpy() if isinstance(a, torch.Tensor) else np.asarray(a)
    p, o = region_params(case), options(case, seed)
    dt, key, N = 0.1, (o["seed"], 0), g.n_neurons
    row_ptr, col, delay = host(g.row_ptr), host(g.col), host(g.delay).astype(np.int64)
    w = (host(g.w_bf16).view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    inh = np.zeros(N, np.int64)
    for r in range(g.n_regions):
        inh[g.region_offsets[r] + g.n_exc[r]:g.region_offsets[r + 1]] = 1
    lam = p["drive_K"] * p["drive_rate_hz"] * dt * 1e-3
    thr, q, cdf = [], math.exp(-lam), math.exp(-lam)
    while len(thr) < 16 and math.floor(cdf * 2.0**32) < 2**32:
        thr.append(math.floor(cdf * 2.0**32))
        q *= lam / len(thr)
        cdf += q
    at = np.arange(-(-N // 4), dtype=np.uint64)
    V = p["Vreset"] + (p["Vth"] - p["Vreset"]) * (philox(0, at, 1, key)[:N] >> np.uint64(40)).astype(np.float64) * 2.0**-24
    J, ref = np.zeros((4, N)), np.zeros(N, np.int64)
    dec = [math.exp(-dt / t) for t in p["tau_u"]]
    n_ref = int(round(p["Tref"] / dt))
    D = int(delay.max()) + 1
    ring = np.zeros((D, 2 * N))
    keys, events = [], 0
    for n in range(case["steps"]):
        u = philox(n, at, 0, key)[:N] >> np.uint64(32)
        a = ring[n % D].reshape(2, N).copy()
        ring[n % D] = 0.0
        for t in thr:
            a[0] += p["w_ext"] * (u >= np.uint64(t))
        current = sum(p["g_u"][c] * J[c] * (p["Vu"][c] - V) for c in range(4)) - p["gL"] * (V - p["VL"]) + p["I_ext"]
        Vn = V + current * dt / p["C"]
        for c in range(4):
            J[c] = dec[c] * J[c] + a[c // 2]
        held = ref > 0
        fired = ~held & (Vn >= p["Vth"])
        V = np.where(held | fired, p["Vreset"], Vn)
        ref = np.where(held, ref - 1, np.where(fired, n_ref, ref))
        for j in np.nonzero(fired)[0]:
            e = slice(row_ptr[j], row_ptr[j + 1])
            np.add.at(ring.reshape(-1), (n + delay[e]) % D * (2 * N) + inh[j] * N + col[e], w[e])
            events += int(row_ptr[j + 1] - row_ptr[j])
            keys.append(n * N + int(j))
    return V, J, ref, np.array(keys, np.int64), events


def exact(case, seed):
    if case["kind"] == "loop":
        V, J, ref, _, _ = simulate64(case, seed, make_graph(case, seed))
        return dict(V=V, J=J, ref=ref, bw=None)
    if case["kind"] == "noalloc":
        V, J, _, _, _ = simulate64(case, seed, make_graph(case, seed, host=False))
        return dict(V=V, J=J, ref=None, spikes=None, events=None)
    return None
