"""One handle used from several threads at once."""
import threading

import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


def _together(jobs):
    """Run the jobs at the same time, each in a thread; raises what one raised."""
    start, errors = threading.Barrier(len(jobs)), []

    def go(job):
        try:
            start.wait()
            job()
        except BaseException as e:      # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=go, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_a_batch_read_by_one_thread_per_instance():
    cfgs = [workload.microcircuit(0.05, seed=90 + k) for k in range(12)]
    stream = torch.cuda.current_stream()
    a, b = (pkg.MicrocircuitBatch(cfgs, stream=stream) for _ in range(2))
    for steps in (400, 30) * 6:
        a.step(steps)
        b.step(steps)
        got = [None] * len(cfgs)

        def read(k):
            got[k] = a.read_spikes(k)

        _together([lambda k=k: read(k) for k in range(len(cfgs))])
        for k in range(len(cfgs)):
            want = b.read_spikes(k)
            np.testing.assert_array_equal(got[k][0], want[0])
            np.testing.assert_array_equal(got[k][1], want[1])
    a.close()
    b.close()


@pytest.mark.parametrize("scale,steps", [(0.1, 7), (1.0, 40)])      # small reads, large ones
def test_a_network_read_while_another_thread_steps_it(scale, steps):
    net, alone = (pkg.Microcircuit(workload.microcircuit(scale), stream=torch.cuda.current_stream()) for _ in range(2))
    buf, parts, stepped = np.empty((2, 1 << 20), np.uint32), [], threading.Event()

    def step():
        for _ in range(150):
            net.step(steps)
        stepped.set()

    def read():
        more = True
        while more:
            more = not stepped.is_set()
            n = net.read_spikes_into(buf[0], buf[1])
            parts.append(buf[:, :n].copy())

    _together([step, read])
    alone.step(150 * steps)
    want = alone.read_spikes()
    got = np.concatenate(parts, axis=1)
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
    net.close()
    alone.close()


def test_a_batch_read_while_another_thread_steps_it():
    cfgs = [workload.microcircuit(0.05, seed=90 + k) for k in range(6)]
    a, b = (pkg.MicrocircuitBatch(cfgs, stream=torch.cuda.current_stream()) for _ in range(2))
    buf, parts, stepped = np.empty((2, 1 << 20), np.uint32), [[] for _ in cfgs], threading.Event()

    def step():
        for _ in range(60):
            a.step(37)
        stepped.set()

    def read():
        more = True
        while more:
            more = not stepped.is_set()
            for k in range(len(cfgs)):
                n = a.read_spikes_into(k, buf[0], buf[1])
                parts[k].append(buf[:, :n].copy())

    _together([step, read])
    b.step(60 * 37)
    for k in range(len(cfgs)):
        got, want = np.concatenate(parts[k], axis=1), b.read_spikes(k)
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])
    a.close()
    b.close()
