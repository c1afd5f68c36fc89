"""The kernels' variants at the sizes where they can go wrong, against the
matched-FP32 oracle, bit for bit: the arithmetic is the oracle's in the same
order and arrivals are exact integers, so the tolerance is zero."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _equal(net, o):
    V, J, r = net.state()
    Vo, Jo, ro = o.state()
    assert np.array_equal(V.astype(np.float64), Vo) and np.array_equal(r, ro)
    assert np.array_equal(J.astype(np.float64), Jo)
    assert np.array_equal(np.stack(net.spikes()), np.stack(o.raster()))
    assert np.allclose(net.bold(), o.bold(), rtol=1e-10, atol=1e-15)
    s, so = net.stats(), o.info()
    assert s["events"] == so["events"] and s["spikes"] == so["spikes"] > 0


# regions that end inside a thread's four neurons, a warp's 128 and a tile's
# 1,024, on their edges, and tiles that lie in one region
@pytest.mark.parametrize("form", ["plain", "current", "two_weights"])
@pytest.mark.parametrize("sizes", [[1021, 6, 1025, 127, 130, 2050], [1024, 2048, 1021], [2051]])
def test_update_region_edges(sizes, form):
    g = synth.make_graph(sizes, 40, 31, k_within=5 if len(sizes) > 1 else 40, d_within=(1, 12), d_cross=(12, 40),
                         region_density=1.0)
    over = dict(ou_mu=0.05, ou_sigma=0.0, ou_tau=8.0, iext_shape=4.0) if form == "current" else {}
    p = [synth.default_region_params(I_ext=0.85 + 0.03 * r, **(over if r != 1 else {})) for r in range(len(sizes))]
    if form == "two_weights":
        g = synth.with_second_weight(g, 5)
    from paper_2211_15963_gb300 import dbnet
    net = dbnet.Network(g, p, dict(seed=6, raster_capacity=1 << 20, tr_ms=5.0))
    o = oracle.Sim(g, p, seed=6, tr_ms=5.0, precision=32)
    net.step(400)
    o.step(400)
    _equal(net, o)
    net.close()


# Every delivery mode on the same spike trains: all edges at emission (small
# ring), windows whose first edges the update adds, windows with the bounds
# ring (forced by a large engine: many members), and one delay per step and
# kernel (the pipelined schedule); step calls that start and end inside
# windows and mix direct steps with replays; longest delays on and off a
# multiple of the window, and shorter than one.
@pytest.mark.parametrize("dmax,bin_ms", [(1, 0.0), (3, 0.0), (8, 0.0), (9, 0.0), (64, 0.0), (255, 0.0), (100, 0.7)])
@pytest.mark.parametrize("schedule", [1, 2, 3])
def test_delivery_modes(dmax, bin_ms, schedule):
    from paper_2211_15963_gb300 import dbnet
    sizes = [1500, 2300, 56_000] if dmax > 9 else [900, 1700]
    g = synth.make_graph(sizes, 40, 7 + dmax, k_within=36, d_within=(1, max(1, dmax // 2)),
                         d_cross=(max(1, dmax // 2), dmax), region_density=1.0)
    p = [synth.default_region_params(I_ext=0.86 + 0.03 * r) for r in range(len(sizes))]
    binned = dict(bin_spikes=1, bin_ms=bin_ms, tr_ms=10 * bin_ms) if bin_ms else dict(tr_ms=10.0)
    net = dbnet.Network(g, p, dict(seed=9, raster_capacity=1 << 20, schedule=schedule, **binned))
    o = oracle.Sim(g, p, seed=9, precision=32, **binned)
    for n in (1, 3, 66, 1, 130, 5, 95):
        net.step(n)
        o.step(n)
        assert net.stats()["events"] == o.info()["events"]
    _equal(net, o)
    net.close()


def test_windows_of_a_large_engine():
    """An ensemble wide enough that its delivery runs in windows with the
    bounds ring and a kernel of its own for the rest of a window: the first,
    a middle and the last member equal single networks (which add every edge
    at emission)."""
    from paper_2211_15963_gb300 import dbnet
    g = synth.make_graph([700, 1100], 60, 3, k_within=48, d_within=(1, 20), d_cross=(20, 75))
    base = [synth.default_region_params(I_ext=0.9)] * 2
    M = 272
    theta = np.random.default_rng(4).uniform(-0.5, 0.5, (M, 2, 2))
    ens = dbnet.Ensemble(g, base, M, theta, dict(seed=8, net_id=40, raster_capacity=1 << 16))
    for n in (5, 300, 1, 94):
        ens.step(n)
    for m in (0, 131, M - 1):
        q = [dict(b) for b in base]
        for r in range(2):
            gu = list(q[r]["g_u"])
            gu[0] *= float(np.exp(theta[m, r, 0]))
            gu[2] *= float(np.exp(theta[m, r, 1]))
            q[r]["g_u"] = tuple(gu)
        net = dbnet.Network(g, q, dict(seed=8, net_id=40 + m, raster_capacity=1 << 16))
        net.step(400)
        for x, y in zip(ens.member_state(m), net.state()):
            assert np.array_equal(x, y)
        a, b = ens.member_spikes(m), net.spikes()
        assert len(b[1]) > 500 and np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        net.close()
    ens.close()


# The resident stepper holds one, two or four tiles a block on up to 16
# blocks, the persistent one a tile a block on one or two blocks an SM: sizes
# on and past each edge, more regions in a tile than a block keeps, every
# form of the update, and calls of one step and of many.
@pytest.mark.parametrize("sizes,form", [([40], "plain"), ([1024], "two_weights"), ([16_000, 384], "plain"),
                                        ([16_385], "current"), ([90] * 30, "plain"), ([90] * 30, "current"),
                                        ([32_768], "two_weights"), ([33_000], "plain"), ([65_536], "current"),
                                        ([66_000], "plain"), ([156_000], "current"), ([100_000, 58_000], "two_weights")])
def test_steppers_that_hold_the_state(sizes, form):
    from paper_2211_15963_gb300 import dbnet
    R = len(sizes)
    k = min(24, sum(sizes) - 1)
    g = synth.make_graph(sizes, k, 17, k_within=max(1, k - 2) if R > 1 else k, d_within=(1, 9), d_cross=(9, 14),
                         region_density=1.0)
    over = dict(ou_mu=0.05, ou_sigma=0.0, ou_tau=8.0, iext_shape=4.0) if form == "current" else {}
    p = [synth.default_region_params(I_ext=0.86 + 0.01 * (r % 5), **(over if r != 1 else {})) for r in range(R)]
    if form == "two_weights":
        g = synth.with_second_weight(g, 5)
    net = dbnet.Network(g, p, dict(seed=6, raster_capacity=1 << 21, tr_ms=5.0))
    assert net.stats()["schedule"] == 3
    o = oracle.Sim(g, p, seed=6, tr_ms=5.0, precision=32)
    for n in (1, 9, 10, 1, 129, 50):
        net.step(n)
        o.step(n)
    _equal(net, o)
    net.close()


def test_noalloc_beyond_the_accumulator_ring():
    """Delays too long for the allocation-free scratch to hold an accumulator
    slot each (40,960 padded neurons x 64 slots): it delivers per step, and
    gives what a handle gives; two steps short of that ring it fits."""
    from paper_2211_15963_gb300 import dbnet
    for n, dmax in ((40_000, 60), (32_000, 62)):
        g = synth.make_graph([n], 30, 23, d_within=(1, dmax))
        p = synth.default_region_params(I_ext=0.9)
        n_pad = -(-n // 1024) * 1024
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        V, J = torch.empty(n_pad, device="cuda"), torch.empty(4, n_pad, device="cuda")
        ref = torch.empty(n_pad, dtype=torch.uint8, device="cuda")
        n_sp, n_ev = dbnet.dbnet_run_noalloc(n, g.region_offsets, g.n_exc, t(g.row_ptr), t(g.col),
                                             t(np.asarray(g.w_bf16).view(np.int16)), t(g.delay), p, dict(seed=4), 250,
                                             V, J, ref)
        net = dbnet.Network(g, p, dict(seed=4))
        net.step(250)
        Vn, Jn, rn = net.state()
        s = net.stats()
        assert n_sp == s["spikes"] > 500 and n_ev == s["events"]
        assert np.array_equal(V[:n].cpu().numpy(), Vn) and np.array_equal(J[:, :n].cpu().numpy(), Jn)
        assert np.array_equal(ref[:n].cpu().numpy(), rn)
        net.close()


@pytest.mark.parametrize("max_neurons,max_delay", [(8_192, 40), (1 << 20, 200)])
def test_server_tunes_with_requests_in_flight(max_neurons, max_delay):
    """A server whose launch shapes are tuned from its first rounds on, while
    requests come and go: its delivery changes from the mode of its size (at
    emission; windows) to per step and back with spikes in flight, and every
    request equals the same network alone."""
    from paper_2211_15963_gb300 import dbnet
    srv = dbnet.Server(max_neurons=max_neurons, max_requests=4, max_regions=16, max_delay=max_delay,
                       chunk_steps=128, arena_bytes=1 << 30, run=dict(autotune_at=64, tr_ms=20.0))
    nets = [synth.make_graph(z, 40, 50 + i, k_within=32 if len(z) > 1 else 40, d_within=(1, 20),
                             d_cross=(20, 40), region_density=1.0)
            for i, z in enumerate(([1500, 700], [2100], [900, 800, 700], [2600, 300]))]
    p = synth.default_region_params(I_ext=0.92)
    todo = [(g, n, i) for i, (g, n) in enumerate(zip(nets * 3, (700, 1500, 1100, 900, 2000, 640, 1300, 800, 1700,
                                                                 1000, 1200, 760)))]
    ids = {srv.submit(g, p, n, seed=30 + i, raster_capacity=1 << 18): (g, n, i) for g, n, i in todo}
    srv.drain()
    for rid, (g, n, i) in ids.items():
        net = dbnet.Network(g, p, dict(seed=30 + i, raster_capacity=1 << 18, tr_ms=20.0, autotune_at=-1))
        net.step(n)
        a, b = srv.spikes(rid), net.spikes()
        assert len(b[1]) > 100 and np.array_equal(np.stack(a), np.stack(b)), i
        assert np.array_equal(srv.bold(rid), net.bold()), i
        net.close()
    srv.close()
