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
    g = synth.make_graph(sizes, 60, 31, k_within=5 if len(sizes) > 1 else 60, d_within=(1, 12), d_cross=(12, 40))
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
