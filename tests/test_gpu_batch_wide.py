"""Batches side by side by the size of their partitions: of fewer neurons than 512
threads, and of more than a CTA has threads (two per thread with the ring in
shared and in global memory, four and eight).  Three networks of one size take
up to 50 partitions each, 150 CTAs, where the batch kernel always takes every
SM: the number of CTAs tells the form."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


# volley: a fifth of one network's neurons start above threshold, more spikes in
# a step than a delivery list or a CTA's shared-memory record holds
@pytest.mark.parametrize("volley", [False, True])
@pytest.mark.parametrize("scale,npt,threads", [
    (0.1, 1, 192), (0.14, 1, 256), (0.2, 1, 352), (0.25, 1, 512),       # small partitions, of fewer threads
    (0.4, 2, 512), (0.6, 2, 512), (0.82, 4, 512), (1.6, 8, 512)])
def test_partitions_match_single_networks(scale, npt, threads, volley):
    cfgs = [workload.microcircuit(scale, seed=60 + k) for k in range(3)]
    cfgs[1] = workload.dc_variant(cfgs[1])
    if volley:
        lo, theta = cfgs[2]["u0_lo"], cfgs[2]["theta"]
        cfgs[2] = dict(cfgs[2], u0_hi=lo + (theta - lo) * 1.25)
    stream = torch.cuda.current_stream()
    batch = pkg.MicrocircuitBatch(cfgs, stream=stream)
    info = batch.info(0)
    assert info["blocks"] == (147 if scale == 0.1 else 150)
    assert info["neurons_per_thread"] == npt and info["threads"] == threads
    got = [[] for _ in cfgs]
    for steps in (1, 2, 47):
        batch.step(steps)
        for k in range(3):
            got[k].append(batch.read_spikes(k))
    batch.sync()
    for k, cfg in enumerate(cfgs):
        net = pkg.Microcircuit(cfg, stream=stream)
        net.step(50)
        st, ids = net.read_spikes()
        assert st.size > (5000 * min(1, scale / 0.4) if volley and k == 2 else 100)
        np.testing.assert_array_equal(np.concatenate([g[0] for g in got[k]]), st)
        np.testing.assert_array_equal(np.concatenate([g[1] for g in got[k]]), ids)
        for a, b in zip(batch.state(k), net.state()):
            np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
        assert batch.counters(k) == net.counters()
        net.close()
    batch.close()


def test_networks_of_two_sizes_in_turns_give_their_own_results():
    """Batches and gradients of a large and a small network, used in turns."""
    stream = torch.cuda.current_stream()
    sizes = ([0.02] * 9, [0.005])
    for tiled in (False, True):
        cfgs = [[workload.microcircuit(s, seed=k) for k, s in enumerate(scales)] for scales in sizes]
        batches = [pkg.MicrocircuitBatch(c, stream=stream) for c in cfgs]
        for b in batches:
            if tiled:
                b.set_tiling(0, 2)
        for which in (0, 1, 0):
            batches[which].step(10)
        for b, c, steps in zip(batches, cfgs, (20, 10)):
            for k, cfg in enumerate(c):
                net = pkg.Microcircuit(cfg, stream=stream, raster_capacity=1 << 16)
                net.step(steps)
                for x, y in zip(b.state(k), net.state()):
                    np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
                net.close()
            b.close()
    nets = [pkg.Microcircuit(workload.microcircuit(s), stream=stream) for s in (0.1, 0.03)]
    turns = [[], []]
    for _ in range(2):
        for k, net in enumerate(nets):
            rates = net.grad_forward(30, 10)
            turns[k].append((rates,) + tuple(net.grad_backward(np.ones(8))))
    for k, s in enumerate((0.1, 0.03)):
        alone = pkg.Microcircuit(workload.microcircuit(s), stream=stream)
        for got in turns[k]:
            rates = alone.grad_forward(30, 10)
            want = (rates,) + tuple(alone.grad_backward(np.ones(8)))
            for x, y in zip(got, want):
                np.testing.assert_array_equal(x, y)
