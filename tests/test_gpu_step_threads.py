"""Networks of few, small partitions: the thread counts on either side of their
lines, in every variant of the step kernel, against the oracle; and several
such networks beside one another on streams of their own."""
import time

import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


@pytest.fixture(scope="module")
def case():
    out = {}
    for heavy in (False, True):         # heavy: inputs that could leave the int32 range
        cfg = dict(workload.microcircuit(0.1), w_scale=300.0 if heavy else 1.0)
        sim = oracle.Simulation(oracle.Network(cfg))
        sim.run(123)
        out[heavy] = cfg, sim.raster(), sim.state(), sim.counters()["saturated"]
    return out


@pytest.mark.parametrize("heavy", [False, True])
@pytest.mark.parametrize("paced", [False, True])
@pytest.mark.parametrize("n_part,most,threads", [
    (64, 121, 192), (41, 189, 192), (40, 193, 256), (31, 249, 256), (30, 258, 352), (22, 351, 352), (21, 368, 512)])
def test_thread_counts(case, n_part, most, threads, paced, heavy):
    cfg, raster, state, saturated = case[heavy]
    net = pkg.Microcircuit(cfg, stream=torch.cuda.current_stream(), n_part=n_part)
    info = net.info()
    assert info["max_part_neurons"] == most and info["threads"] == threads
    assert info["saturation_check"] == int(heavy)
    if paced:
        net.set_realtime(1000)
    for steps in (1, 2, 120):
        net.step(steps)
    if saturated:
        with pytest.raises(pkg.SnnError) as e:
            net.sync()
        assert e.value.code == pkg.SNN_ERR_SATURATED
    else:
        net.sync()
    got = net.read_spikes()
    assert raster[0].size > 100
    np.testing.assert_array_equal(got[0], raster[0])
    np.testing.assert_array_equal(got[1], raster[1])
    for g, o in zip(net.state(), state):
        np.testing.assert_array_equal(g.view(np.uint32), o.view(np.uint32))
    np.testing.assert_array_equal(net.ring(), state[3].astype(np.int32))


def test_networks_on_streams_of_their_own_run_beside_one_another():
    """Nine networks of 10 % take about as long as one (twice, where the machine
    holds them back); in turns they would take three times as long and more."""
    nets = [pkg.Microcircuit(workload.microcircuit(0.1, 5 + k), stream=torch.cuda.Stream(), raster_capacity=1 << 20)
            for k in range(9)]

    def seconds(some):
        best = 1e9
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for net in some:
                net.step(2000)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best

    one, all_nine = seconds(nets[:1]), seconds(nets)
    assert all_nine < 2.0 * one, (one, all_nine)
    for net, k in ((nets[0], 0), (nets[8], 8)):
        alone = pkg.Microcircuit(workload.microcircuit(0.1, 5 + k), stream=torch.cuda.current_stream())
        alone.step(net.counters()["step"])
        assert alone.counters() == net.counters()
        for a, b in zip(alone.state(), net.state()):
            np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
