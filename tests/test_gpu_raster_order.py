"""The raster reads come sorted by (step, id): few and many spikes, steps with
more spikes than one warp ranks, spans with more steps than buckets, steps
recorded twice after a restored state, and reads shorter than the raster."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


def _net(scale, n_above=0, **kw):
    cfg = workload.microcircuit(scale)
    u0 = workload.transient_membrane(cfg, seed=9, n_above=n_above) if n_above else None
    return pkg.Microcircuit(cfg, u0=u0, stream=torch.cuda.current_stream(), **kw)


def _pieces(net, chunks):
    """The raster read after every chunk: sorted pieces of ascending steps."""
    out = []
    for c in chunks:
        net.step(c)
        out.append(net.read_spikes())
    return np.concatenate([p[0] for p in out]), np.concatenate([p[1] for p in out])


@pytest.mark.parametrize("scale,n_above,steps", [
    (0.02, 0, 3), (0.1, 0, 40), (0.1, 0, 1500), (0.1, 3000, 2), (0.1, 600, 300), (1.0, 20000, 60)])
def test_one_read_equals_reads_step_by_step(scale, n_above, steps):
    a, b = _net(scale, n_above), _net(scale, n_above)
    a.step(steps)
    st, ids = a.read_spikes()
    assert st.size == a.counters()["spikes"] and st.dtype == ids.dtype == np.int64
    key = st << 20 | ids
    assert np.all(key[1:] > key[:-1])
    chunks = [1] * min(steps, 60) + ([steps - 60] if steps > 60 else [])
    w_st, w_id = _pieces(b, chunks)
    np.testing.assert_array_equal(st, w_st)
    np.testing.assert_array_equal(ids, w_id)


def test_more_steps_than_buckets():
    a, b = _net(0.001), _net(0.001)
    steps = (1 << 20) * 2 + 77
    a.step(steps)
    st, ids = a.read_spikes()
    assert st.size > 2048 and st[-1] > 1 << 20
    w_st, w_id = _pieces(b, [steps // 5] * 5 + [steps % 5])
    np.testing.assert_array_equal(st, w_st)
    np.testing.assert_array_equal(ids, w_id)


def test_steps_recorded_twice_and_short_reads():
    net = _net(0.1, 1500)
    start = net.save_state()
    net.step(80)
    once = net.read_spikes()
    net.load_state(start)
    net.step(80)
    net.load_state(start)
    net.step(30)
    first = once[0] < 30
    want = np.concatenate([once[0], once[0][first]]), np.concatenate([once[1], once[1][first]])
    order = np.lexsort((want[1], want[0]))
    st, ids = net.read_spikes()
    np.testing.assert_array_equal(st, want[0][order])
    np.testing.assert_array_equal(ids, want[1][order])
    net.load_state(start)
    net.step(80)
    buf = np.zeros((2, 1700), np.uint32)
    with pytest.raises(pkg.SnnError):
        net.read_spikes_into(buf[0], buf[1])
    np.testing.assert_array_equal(buf[0], once[0][:1700])
    np.testing.assert_array_equal(buf[1], once[1][:1700])


def test_batch_reads_are_sorted():
    cfgs = [workload.microcircuit(s, seed=40 + k) for k, s in enumerate((0.03, 0.011, 0.05))]
    batch = pkg.MicrocircuitBatch(cfgs, stream=torch.cuda.current_stream())
    got = [[], [], []]
    for steps, reads in ((3, (1,)), (700, (0, 1, 2)), (1200, (2, 0)), (5, (0, 1, 2))):
        batch.step(steps)
        for k in reads:
            got[k].append(batch.read_spikes(k))
    for k, cfg in enumerate(cfgs):
        net = pkg.Microcircuit(cfg, stream=torch.cuda.current_stream())
        net.step(1908)
        st, ids = net.read_spikes()
        np.testing.assert_array_equal(np.concatenate([g[0] for g in got[k]]), st)
        np.testing.assert_array_equal(np.concatenate([g[1] for g in got[k]]), ids)


def test_reads_from_several_threads():
    """One handle read from several threads at once: every read is whole."""
    import threading

    net = _net(0.05)
    net.step(300)
    net.sync()
    want, counts, ring = net.state(), net.counters(), net.ring()
    wrong = []

    def read(kind):
        for _ in range(60):
            if kind == 0:
                ok = all(np.array_equal(a.view(np.uint32), b.view(np.uint32)) for a, b in zip(net.state(), want))
            elif kind == 1:
                ok = net.counters() == counts and net.raster_size() == counts["spikes"]
            else:
                ok = np.array_equal(net.ring(), ring)
            if not ok:
                wrong.append(kind)

    threads = [threading.Thread(target=read, args=(k % 3,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
