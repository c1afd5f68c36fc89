"""Delivery modes and launch shapes at the edges of the rules that choose
them: against the matched-FP32 oracle, or against another mode of the same
network.  The arithmetic is the same in the same order and arrivals are exact
integers, so the tolerance is zero."""
import threading

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


def _net(g, p, **opts):
    from paper_2211_15963_gb300 import dbnet
    return dbnet.Network(g, p, opts)


def _same(net, other):
    for a, b in zip(net.state(), other.state()):
        assert np.array_equal(np.asarray(a, np.float64), np.asarray(b, np.float64))


# Windows on networks whose longest delay is below, at and just above a
# window's eight steps: the accumulators of every delay at once (a power of two
# of slots, 8 bytes a neuron, 16 with two weights) lie beyond the emission
# ring's 48 MB; the update adds the edges due in the window (up to 532 tiles)
# or a kernel of its own does, with two weights and with one.
@pytest.mark.parametrize("n,dmax,two", [(400_000, 5, True), (400_000, 6, True), (400_000, 7, True), (200_000, 8, True),
                                        (200_000, 9, True), (1_600_000, 1, True), (800_000, 3, True),
                                        (1_600_000, 3, False)])
def test_windows_and_short_delays(n, dmax, two):
    g = synth.make_graph([n // 2, n - n // 2], 20, 5, k_within=16, d_within=(1, dmax), d_cross=(1, dmax))
    assert g.delay.max() == dmax
    if two:
        g = synth.with_second_weight(g, 5)
    p = [synth.default_region_params(I_ext=0.88 + 0.03 * r) for r in range(2)]
    net = _net(g, p, seed=3, tr_ms=5.0)
    o = oracle.Sim(g, p, seed=3, tr_ms=5.0, precision=32)
    for k in (1, 6, 66, 3, 9):
        net.step(k)
        o.step(k)
        s, so = net.stats(), o.info()
        assert s["events"] == so["events"] and s["spikes"] == so["spikes"] > 0, k
    _same(net, o)
    net.close()


def test_persistent_schedule_on_more_tiles_than_blocks():
    """The persistent schedule by option on more tiles than its blocks: each
    block takes several tiles of a step, in windows with their own kernel's
    part for the rest of a window.  The autotuner has nothing to weigh there;
    the schedule stays what the options say and nothing fails."""
    g = synth.make_graph([300_000, 400_000], 10, 11, k_within=8, d_within=(1, 12), d_cross=(12, 60))
    p = [synth.default_region_params(I_ext=0.88 + 0.03 * r) for r in range(2)]
    net = _net(g, p, seed=5, schedule=3, autotune_at=64)
    plain = _net(g, p, seed=5, schedule=1, autotune_at=-1)
    for n in (30, 100, 130):
        net.step(n)
        plain.step(n)
        _same(net, plain)
        s, sp = net.stats(), plain.stats()
        assert s["schedule"] == 3 and s["events"] == sp["events"] and s["spikes"] == sp["spikes"] > 0
    assert s["autotuned"] == 1
    net.close()
    plain.close()


def test_a_losing_rule_is_left_with_binned_spikes():
    """60,000 neurons at some 800,000 events a step, far above what one
    cluster's SMs reduce: the resident stepper takes twice the time of the
    best per-step shape, and the tuner's verdict to leave it holds although
    its turns end inside a bin."""
    k = 1000
    g = synth.make_graph([30_000, 30_000], k, 27, k_within=800, d_within=(1, 10), d_cross=(10, 20))
    p = synth.default_region_params(I_ext=97.0)
    p["g_u"] = tuple(x * 100.0 / k for x in p["g_u"])
    opts = dict(seed=4, bin_spikes=1)
    rule = _net(g, p, autotune_at=-1, **opts)
    net = _net(g, p, autotune_at=64, **opts)
    net.step(6000)
    rule.step(6000)
    s, r = net.stats(), rule.stats()
    assert s["events"] == r["events"] > 6000 * 500_000 and s["autotuned"] == 1
    assert r["schedule"] == 3 and s["deliver_blocks"] != r["deliver_blocks"]  # of a per-step shape
    for a, b in zip(net.state(), rule.state()):
        assert np.array_equal(a, b)
    net.close()
    rule.close()


def test_calls_shorter_than_a_tuning_turn():
    """A program that stops in the middle of the tuning and goes on with
    calls too short for a turn steps in the mode of the engine's size, not
    in the candidate that came last; longer calls finish the tuning."""
    g = synth.small_network()
    p = synth.default_region_params()
    net = _net(g, p, seed=7, autotune_at=64, raster_capacity=1 << 20)
    o = oracle.Sim(g, p, seed=7, precision=32)
    for n in (64 + 64, 10, 1, 9, 200, 63, 64, 10):
        net.step(n)
        o.step(n)
        s = net.stats()
        if n < 64:
            assert s["schedule"] == 3 and s["autotuned"] == 0
        assert s["events"] == o.info()["events"]
        _same(net, o)
    for n in (5000, 10, 2000):
        net.step(n)
        o.step(n)
    assert net.stats()["autotuned"] == 1 and net.stats()["events"] == o.info()["events"]
    assert np.array_equal(np.stack(net.spikes()), np.stack(o.raster()))
    _same(net, o)
    net.close()


# More regions than the warps of one block close at once, on one block and on
# sixteen, closing every step and every tenth.
@pytest.mark.parametrize("size,regions,dt", [(4, 1000, 0.1), (5, 1300, 1.0), (40, 1200, 0.1)])
def test_many_regions_on_the_resident_stepper(size, regions, dt):
    g = synth.make_graph([size] * regions, 20, 19, k_within=2, d_within=(1, 3), d_cross=(1, 9))
    p = [synth.default_region_params(I_ext=0.86 + 0.01 * (r % 5)) for r in range(regions)]
    over = dict(dt_ms=dt, bin_ms=1.0, tr_ms=2.0)
    net = _net(g, p, seed=6, **over)
    assert net.stats()["schedule"] == 3
    o = oracle.Sim(g, p, seed=6, precision=32, **over)
    for n in (1, 39, 60):
        net.step(n)
        o.step(n)
    _same(net, o)
    assert len(net.bold()) > 0 and np.allclose(net.bold(), o.bold(), rtol=1e-10, atol=1e-15)
    net.close()


@pytest.mark.parametrize("schedule", [1, 2, 3])
def test_emission_threshold_with_a_ring_of_any_length(schedule):
    """An explicit emission threshold is kept wherever a slot per step of the
    longest delay fits a third of the free memory, also where the next power
    of two of slots does not."""
    n, dmax = 1_000_000, 128
    g = synth.make_graph([n // 2, n - n // 2], 10, 13, k_within=8, d_within=(1, 20), d_cross=(20, dmax))
    p = [synth.default_region_params(I_ext=0.88 + 0.03 * r) for r in range(2)]
    plain = _net(g, p, seed=9, schedule=2, autotune_at=-1)
    plain.step(200)
    state, events = plain.state(), plain.stats()["events"]
    plain.close()
    torch.cuda.empty_cache()
    slot = -(-n // 1024) * 1024 * 8
    need = int(4.2 * (dmax + 1) * slot)  # a third of this holds 129 slots, not 256
    hold = torch.empty(torch.cuda.mem_get_info()[0] - need, dtype=torch.uint8, device="cuda")
    try:
        net = _net(g, p, seed=9, emit_delay=30, autotune_at=-1, schedule=schedule)
        for k in (1, 70, 129):
            net.step(k)
        assert net.stats()["emit_delay"] == 30
        for a, b in zip(net.state(), state):
            assert np.array_equal(a, b)
        assert net.stats()["events"] == events
        net.close()
    finally:
        del hold
        torch.cuda.empty_cache()


def test_one_segment_ring():
    """An engine that delivers in windows and may be tuned holds one segment
    ring, not one for the windows and one for the tuner's per-step turns."""
    g = synth.make_graph([600_000], 10, 15, d_within=(1, 200))
    p = synth.default_region_params(I_ext=0.9)

    def held(**opts):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        net = _net(g, p, seed=2, **opts)
        used = before - torch.cuda.mem_get_info()[0]
        for n in (300, 4000, 100):
            net.step(n)
        state = net.state()
        net.close()
        return used, state

    held(schedule=2)  # what the first use of each path takes once
    held(autotune_at=128)
    per_step, a = held(schedule=2, autotune_at=-1)
    windows, b = held(autotune_at=128)
    # the ring alone: a 64th of the neurons x 204 slots x 51 bounds of 2 bytes
    assert windows - per_step < 9376 * 204 * 51 * 2 // 2
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_persistent_networks_on_two_threads():
    """Two networks on the persistent stepper, stepped at the same time from
    two threads, each with a grid that fills the device: their launches take
    turns, no barrier gives up, and each equals the same network alone."""
    p = synth.default_region_params(I_ext=0.9)
    nets, alone = [], []
    for k in range(2):
        g = synth.make_graph([290_000], 10, 21 + k, d_within=(1, 60))
        a = _net(g, p, seed=30 + k, autotune_at=-1)
        a.step(600)
        alone.append((a.state(), a.stats()["events"]))
        a.close()
        nets.append(_net(g, p, seed=30 + k, autotune_at=-1))
        assert nets[k].stats()["schedule"] == 3
    failed = []

    def run(net):
        try:
            for n in (1, 99, 300, 200):
                net.step(n)
            net.sync()
        except Exception as e:  # noqa: BLE001 (reported below)
            failed.append(e)

    th = [threading.Thread(target=run, args=(net,)) for net in nets]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not failed, failed
    for net, (state, events) in zip(nets, alone):
        for x, y in zip(net.state(), state):
            assert np.array_equal(x, y)
        assert net.stats()["events"] == events
        net.close()


@pytest.mark.parametrize("max_neurons,max_delay,tune_at", [(8_192, 40, -1), (8_192, 40, 64), (200_000, 200, 64)])
def test_server_on_the_persistent_schedule(max_neurons, max_delay, tune_at):
    """A server by option on the persistent stepper, whose blocks hold their
    tiles' state and constants: short requests of several regions come and
    go, so that graphs and constants of finished ones pass to others while
    launches are in flight.  Every request equals the same network alone."""
    from paper_2211_15963_gb300 import dbnet
    p = synth.default_region_params(I_ext=0.92)
    nets = [synth.make_graph(z, 40, 50 + i, k_within=32 if len(z) > 1 else 40, d_within=(1, 20), d_cross=(20, 40),
                             region_density=1.0)
            for i, z in enumerate(([1500, 700], [2100], [900, 800, 700], [100] * 12))]
    srv = dbnet.Server(max_neurons=max_neurons, max_requests=4, max_regions=40, max_delay=max_delay, chunk_steps=100,
                       arena_bytes=1 << 29, run=dict(autotune_at=tune_at, tr_ms=20.0, schedule=3))
    todo = [(k % 4, 150 + 137 * ((5 * k) % 11), k) for k in range(24)]
    ids = {srv.submit(nets[j], p, n, seed=30 + i, raster_capacity=1 << 18): (j, n, i) for j, n, i in todo}
    srv.drain()
    for rid, (j, n, i) in ids.items():
        net = _net(nets[j], p, seed=30 + i, raster_capacity=1 << 18, tr_ms=20.0, autotune_at=-1, schedule=2)
        net.step(n)
        a, b = srv.spikes(rid), net.spikes()
        assert len(b[1]) > 100 and np.array_equal(np.stack(a), np.stack(b)), i
        assert np.array_equal(srv.bold(rid), net.bold()), i
        net.close()
    srv.close()


def test_windows_of_one_step():
    """Two steps' accumulators beyond the L2: windows of one step on one
    accumulator slot, whose bounds ring keeps a bound for every delay, against
    per-step delivery, through the tuner and back."""
    g = synth.make_graph([4_700_000, 4_900_000], 4, 29, k_within=3, d_within=(1, 5), d_cross=(5, 11))
    p = [synth.default_region_params(I_ext=0.9 + 0.03 * r) for r in range(2)]
    net = _net(g, p, seed=3, autotune_at=90)
    plain = _net(g, p, seed=3, schedule=2, autotune_at=-1)
    for n in (1, 2, 70, 17, 300, 20, 2500):
        net.step(n)
        plain.step(n)
        s, sp = net.stats(), plain.stats()
        assert s["events"] == sp["events"] and s["spikes"] == sp["spikes"] > 0
    _same(net, plain)
    net.close()
    plain.close()
