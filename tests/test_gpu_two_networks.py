"""Networks, gradients and batches of different sizes made one after the other
and used in turn: the later, smaller one must not take the earlier one's
shared memory away."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


def test_networks_of_two_sizes_take_turns():
    stream = torch.cuda.current_stream()
    nets = [pkg.Microcircuit(workload.microcircuit(s), stream=stream) for s in (0.9, 0.7, 0.1, 0.05)]
    for _ in range(2):
        for net in nets:
            net.step(20)
            net.sync()
    for net, s in zip(nets, (0.9, 0.7, 0.1, 0.05)):
        alone = pkg.Microcircuit(workload.microcircuit(s), stream=stream)
        alone.step(40)
        np.testing.assert_array_equal(net.state()[0].view(np.uint32), alone.state()[0].view(np.uint32))


def test_gradients_of_two_sizes_take_turns():
    stream = torch.cuda.current_stream()
    nets = [pkg.Microcircuit(workload.microcircuit(s), stream=stream) for s in (0.1, 0.03)]
    out = []
    for _ in range(2):
        for net in nets:
            net.grad_forward(30, 10)
            out.append(net.grad_backward(np.ones(8))[0])
    assert all(np.abs(g).max() > 0 for g in out)


def test_batches_of_two_sizes_take_turns():
    stream = torch.cuda.current_stream()
    big = pkg.MicrocircuitBatch([workload.microcircuit(0.02, seed=k) for k in range(9)], stream=stream)
    small = pkg.MicrocircuitBatch([workload.microcircuit(0.005, seed=3)], stream=stream)
    for tiled in (False, True):
        for b in (big, small):
            if tiled:
                b.set_tiling(0, 2)
        for b in (big, small, big):
            b.step(10)
            b.sync()
