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
