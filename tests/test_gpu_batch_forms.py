"""A batch whose instances fit on the GPU side by side runs as partitions of
their own (no barrier over the batch); asking for a tiling takes it on to the
batch kernel.  Every instance against a single network of its own, bit for
bit, in both forms and across the change."""
import copy

import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


def _check(batch, cfgs, steps, reads):
    for k, cfg in enumerate(cfgs):
        net = pkg.Microcircuit(cfg, stream=torch.cuda.current_stream())
        net.step(steps)
        st, ids = net.read_spikes()
        assert st.size > 0 or workload.n_neurons(cfg) < 100
        got = reads[k] + [batch.read_spikes(k)]
        np.testing.assert_array_equal(np.concatenate([g[0] for g in got]), st)
        np.testing.assert_array_equal(np.concatenate([g[1] for g in got]), ids)
        for a, b in zip(batch.state(k), net.state()):
            np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
        c, d = batch.counters(k), net.counters()
        assert c == d


@pytest.mark.parametrize("scales,npt", [
    ((0.0004,), 1),                             # one partition of 31 neurons
    ((0.03, 0.0123, 0.05, 0.007, 0.021), 1),
    ((0.3, 0.5, 0.111), 1),                     # nearly every SM
    ((0.9, 0.4, 0.7), 2),                       # ring in shared memory, two neurons per thread
    ((1.3, 0.6), 2),                            # ring in global memory
])
def test_partitioned_batch_matches_single_networks(scales, npt):
    cfgs = [workload.microcircuit(s, seed=70 + k) for k, s in enumerate(scales)]
    if len(cfgs) > 2:
        cfgs[2] = workload.dc_variant(cfgs[2])
    batch = pkg.MicrocircuitBatch(cfgs, stream=torch.cuda.current_stream())
    info = batch.info(0)
    if npt == 1:
        assert info["neurons_per_thread"] == 1 and info["blocks"] <= 152
    reads = [[] for _ in cfgs]
    for n in (1, 6, 50):
        batch.step(n)
        reads[0].append(batch.read_spikes(0))
    batch.sync()
    _check(batch, cfgs, 57, reads)
    batch.close()


@pytest.mark.parametrize("before", [3, 1000, 1061])
def test_tiling_asked_for_in_mid_run(before):
    cfgs = [workload.microcircuit(s, seed=80 + k) for k, s in enumerate((0.03, 0.011, 0.02))]
    batch = pkg.MicrocircuitBatch(cfgs, stream=torch.cuda.current_stream())
    batch.step(before)
    reads = [[], [batch.read_spikes(1)], []]
    batch.step(2)
    batch.set_tiling(1, 1)
    batch.set_tiling(0, 0)
    assert batch.info(1)["tiling"] == 1
    batch.step(1003)
    batch.sync()
    _check(batch, cfgs, before + 1005, reads)
    batch.close()


# 267,703 spikes (the oracle's count), all of one partition, whose list holds 262,144
@pytest.mark.parametrize("capacity,fits", [(267_703, True), (267_702, False)])
def test_one_partition_may_use_the_whole_capacity(capacity, fits):
    hot = copy.deepcopy(workload.dc_variant(workload.microcircuit(0.002)))
    hot["i_dc"] = [20000.0] * 8
    cold = copy.deepcopy(workload.dc_variant(workload.microcircuit(0.008)))
    cold["i_dc"] = [0.0] * 8
    cfgs = [cold, hot, cold, cold, cold]
    batch = pkg.MicrocircuitBatch(cfgs, stream=torch.cuda.current_stream(), raster_capacity=capacity)
    assert batch.info(0)["neurons_per_thread"] == 1
    net = pkg.Microcircuit(hot, stream=torch.cuda.current_stream())
    batch.step(90_000)
    net.step(90_000)
    st, ids = net.read_spikes()
    assert st.size == 267_703
    if fits:
        batch.sync()
        got = batch.read_spikes(1)
        np.testing.assert_array_equal(got[0], st)
        np.testing.assert_array_equal(got[1], ids)
    else:
        for call in (batch.sync, lambda: batch.read_spikes(1)):
            with pytest.raises(pkg.SnnError) as e:
                call()
            assert e.value.code == pkg.SNN_ERR_OVERFLOW
    batch.close()
