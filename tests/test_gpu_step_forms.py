"""The forms of the step kernel on either side of the lines between them: the
spike count published ahead of the CTA barrier (at most 64 partitions, several
neurons per thread) or at it, launches of one and two steps and of many, and
lists longer than the message heads hold."""
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
    cfg = workload.microcircuit(0.1)
    sim = oracle.Simulation(oracle.Network(cfg))
    sim.run(204)
    return cfg, sim.raster(), sim.state()


# 3 and 15 partitions: six and two neurons per thread
@pytest.mark.parametrize("n_part", [3, 15, 64, 65, 152])
def test_launches_of_any_length_on_either_side(case, n_part):
    cfg, raster, state = case
    net = pkg.Microcircuit(cfg, stream=torch.cuda.current_stream(), n_part=n_part)
    for steps in (1, 1, 2, 200):
        net.step(steps)
    got = net.read_spikes()
    assert raster[0].size > 100
    np.testing.assert_array_equal(got[0], raster[0])
    np.testing.assert_array_equal(got[1], raster[1])
    for g, o in zip(net.state(), state):
        np.testing.assert_array_equal(g.view(np.uint32), o.view(np.uint32))
    np.testing.assert_array_equal(net.ring(), state[3].astype(np.int32))
