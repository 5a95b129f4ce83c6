"""What the library's host code asks of the CUDA runtime, seen without a GPU:
the library runs in a child process on a runtime whose kernels do nothing
(host/fake_cudart.cpp) and the test reads the log of the calls."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda"

PRELUDE = """
import ctypes, re, sys
sys.path.insert(0, {root!r})
rt = ctypes.CDLL("libcudart.so.13")
rt.fake_log.restype = ctypes.c_char_p
rt.fake_alloc_limit.argtypes = [ctypes.c_size_t]
rt.fake_alloc.restype = ctypes.c_void_p
rt.fake_alloc.argtypes = [ctypes.c_size_t, ctypes.c_int]
rt.fake_raster_count.restype = ctypes.POINTER(ctypes.c_uint32)
import numpy as np
import paper_1909_08665_gb300 as pkg
import workload


def words(n, k=0):
    # the k-th device array of n 32-bit words
    return np.ctypeslib.as_array(ctypes.cast(rt.fake_alloc(4 * n, k), ctypes.POINTER(ctypes.c_uint32)), (n,))


def calls(kind):
    return [x for x in rt.fake_log().decode().splitlines() if x.split()[0] == kind]


class Stream:
    cuda_stream = 0x40

"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(CUDA + "/include/cuda_runtime_api.h"):
        pytest.skip("needs g++ and the CUDA headers")
    from paper_1909_08665_gb300 import _build
    _build.build()
    d = tmp_path_factory.mktemp("cudart")
    (d / "version").write_text("libcudart.so.13 { global: *; };\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CUDA + "/include",
                    os.path.join(ROOT, "tests", "host", "fake_cudart.cpp"), "-o", str(d / "libcudart.so.13"),
                    "-Wl,-soname,libcudart.so.13", "-Wl,--version-script," + str(d / "version")], check=True)

    def go(body):
        env = dict(os.environ, LD_LIBRARY_PATH=str(d) + ":" + os.environ.get("LD_LIBRARY_PATH", ""))
        r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + body], env=env, capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout
    return go


def test_batch_steps_do_not_wait(run):
    """A batch side by side steps on its stream whatever the number of steps."""
    run("""
b = pkg.MicrocircuitBatch([workload.microcircuit(s) for s in (0.03, 0.0123, 0.05)], stream=Stream())
assert b.info(0)["neurons_per_thread"] == 1
rt.fake_clear()
b.step(50_321)
assert len(calls("graph")) == 50 and calls("launch") and not calls("sync"), rt.fake_log()
""")


def test_batch_raster_is_as_large_as_asked_for(run):
    """Two arrays of the capacity, and nothing larger."""
    run("""
for cap in (0, 4 << 20, 65 << 20):
    rt.fake_clear()
    b = pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 3, stream=Stream(), raster_capacity=cap)
    sizes = sorted(int(x.split()[-1]) for x in calls("malloc"))
    assert sizes[-2:] == [4 * (cap or 64 << 20)] * 2 and sizes[-3] < 16 << 20, (cap, sizes[-4:])
    b.close()
""")


def test_a_larger_raster_capacity_never_shortens_a_list(run):
    """A partition's list is the share of a partition of 512 neurons (of all
    neurons in few), until the lists take the default's memory."""
    run("""
for scale in (0.005, 0.1, 0.3, 1.0):
    need = -(-workload.n_neurons(workload.microcircuit(scale)) // 512)
    last = 0
    for cap in (1 << 20, 12 << 20, 40 << 20, 64 << 20, 0, 65 << 20, 200 << 20):
        rt.fake_clear()
        net = pkg.Microcircuit(workload.microcircuit(scale), stream=Stream(), raster_capacity=cap)
        sizes = [int(x.split()[-1]) for x in calls("malloc")]
        asked, parts = cap or 64 << 20, net.info()["n_part"]
        entries = min(asked // min(need, 152), max(asked, 64 << 20) // parts)
        assert sizes.count(4 * entries * parts) == 2 and entries >= max(last, asked // parts), (scale, cap, sorted(sizes)[-4:])
        last = entries
        net.close()
""")


def test_batch_spikes_read_by_two_threads(run):
    """A read that finds the raster drained waits until another thread's drain
    has handed the spikes out."""
    run("""
import threading, time
n = 3_000_000
b = pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 2, stream=Stream())
b.step(1)
b.read_spikes(0)
bufs = [np.empty((2, n), np.uint32) for _ in range(2)]
rt.fake_raster_count()[0] = n
b.step(1)
b.read_spikes_into(0, *bufs[0])             # makes the arrays the sorted spikes lie in
for delay in range(200):                    # at every stage of the other's drain
    b.step(1)
    rt.fake_raster_count()[0] = n           # all of instance 0
    words(n, 0)[:] = words(n, 1)[:] = delay
    got, done = [0, 0], threading.Event()

    def drain():
        got[1] = b.read_spikes_into(1, *bufs[1])
        done.set()

    t = threading.Thread(target=drain)
    t.start()
    time.sleep(delay * 1.25e-4)
    while not done.is_set():
        got[0] += b.read_spikes_into(0, *bufs[0])
    t.join()
    got[0] += b.read_spikes_into(0, *bufs[0])
    assert got == [n, 0] and (bufs[0] == delay).all(), (delay, got)
""")


def test_reads_work_from_another_device(run):
    """A handle's reads launch and allocate on its own device, whichever one is
    current, and leave that current."""
    run("""
net = pkg.Microcircuit(workload.microcircuit(0.02), stream=Stream())
large = pkg.Microcircuit(workload.microcircuit(0.5), stream=Stream())
b = pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 2, stream=Stream())
many = [np.empty(5000, np.uint32) for _ in range(2)]
for h, read in ((net, lambda: net.read_spikes_into(*many)), (b, lambda: b.read_spikes_into(1, *many))):
    h.step(3)
    read()
    rt.fake_raster_count()[0] = 5000         # sorted on the device by the next read
    h.step(3)
    for call in (read, net.raster_size, net.counters, net.ring, net.state, large.state,
                 lambda: net.load_state(net.save_state()), lambda: b.state(1), lambda: b.counters(0)):
        rt.fake_set_device(1)
        rt.fake_clear()
        call()
        assert rt.fake_device() == 1
        assert not [x for x in calls("launch") + calls("malloc") if " dev 0" not in x], rt.fake_log()
        rt.fake_set_device(0)
""")


def test_raster_reads_without_device_memory(run):
    """Where the device has no room for the sort's arrays the spikes come
    sorted all the same."""
    run("""
n, cap = 5000, 77_777
rng = np.random.default_rng(3)
net = pkg.Microcircuit(workload.microcircuit(0.02), stream=Stream(), raster_capacity=cap, n_part=1)
b = pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 3, stream=Stream(), raster_capacity=cap + 1)
one = workload.n_neurons(workload.microcircuit(0.02))
for h, total, entries in ((net, one, cap), (b, 3 * one, cap + 1)):
    h.step(100)
    read = h.read_spikes_into if h is net else (lambda s, i: h.read_spikes_into(1, s, i))
    buf = np.zeros((2, n), np.uint32)
    read(*buf)
    h.step(100)
    rt.fake_raster_count()[0] = n
    st, ids = words(entries, 0), words(entries, 1)
    st[:n], ids[:n] = rng.integers(100, 200, n), rng.integers(0, total, n)
    rt.fake_alloc_limit(1 << 12)
    got = read(*buf)
    rt.fake_alloc_limit(1 << 40)
    st, ids = st[:n], ids[:n]
    if h is b:
        mine = (ids >= one) & (ids < 2 * one)
        st, ids = st[mine], ids[mine] - one
    order = np.lexsort((ids, st))
    assert got == st.size > 1000
    assert (buf[0, :got] == st[order]).all() and (buf[1, :got] == ids[order]).all()
    h.step(100)
    rt.fake_raster_count()[0] = n            # a short read keeps the first ones
    if h is net:
        st[:] = 100 + st
        rt.fake_alloc_limit(1 << 12)
        try:
            net.read_spikes_into(buf[0, :100], buf[1, :100])
            assert False
        except pkg.SnnError as e:
            assert e.code == pkg.SNN_ERR_OVERFLOW
        rt.fake_alloc_limit(1 << 40)
        assert (buf[0, :100] == np.sort(st)[:100]).all()
""")


def test_gradients_near_the_shared_memory_limit_stay_partition_local(run):
    """The largest network whose rows fit beside the window and the tables: the
    flags of its spikes take no room of their own."""
    run("""
import oracle


def adjoint_kernel(scale):
    # the kernel the backward of a network of this scale launches
    cfg = workload.microcircuit(scale)
    rp, tg, dl, code = oracle.Network(cfg).export()
    n = rp.size - 1
    parts = -(-n // 512)
    lo = np.arange(parts + 1) * n // parts
    ncmax = int(np.diff(lo).max())
    packed = tg.astype(np.uint32) | dl.astype(np.uint32) << 19 | code.astype(np.uint32) << 25
    wtab = np.ones((8, 8, 128), np.int32)
    net = pkg.Microcircuit(cfg, stream=Stream(), n_part=parts, raster_capacity=1 << 16,
                           rows={"row_ptr": rp, "words": packed, "wtab": wtab})
    # what the kernels would have made of the rows: every partition's run, and
    # the entries the step kernel reads
    src = np.repeat(np.arange(n), np.diff(rp))
    at = np.searchsorted(src * n + tg, (np.arange(n)[:, None] * n + lo[None]).ravel()).astype(np.uint32)
    words(n * (parts + 1) + 4)[:at.size] = at
    pop = np.repeat(np.arange(8), cfg["pop_sizes"])
    part = np.searchsorted(lo, tg, side="right") - 1
    index = (pop[tg] * 8 + pop[src]) * 128 + code
    words(tg.size + 4, 1)[:tg.size] = index.astype(np.uint32) << 19 | (dl.astype(np.uint32) * ncmax + (tg - lo[part]).astype(np.uint32))
    net.grad_forward(20, 10)
    rt.fake_clear()
    net.grad_backward(np.ones(8))
    names = [x.split()[1] for x in calls("launch") if "k_adjoint" in x and "fold" not in x]
    net.close()
    return names[-1]


assert "k_adjoint_part" in adjoint_kernel(0.102)
""")


def test_shared_memory_limits_are_never_lowered(run):
    """A kernel's limit belongs to the whole process: whichever network sets it,
    it is the most a block may have."""
    run("""
nets = [pkg.Microcircuit(workload.microcircuit(s), stream=Stream(), raster_capacity=1 << 16) for s in (0.3, 0.02)]
spikes = np.zeros(8, np.uint32)
for net in nets:
    for tiling in (2, 3, 4, 5):
        net.deliver(spikes.ctypes.data, 8, 0, tiling)
    net.grad_forward(4, 2)
    net.grad_backward(np.ones(8))
b = pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 3, stream=Stream(), raster_capacity=1 << 16)
b.set_tiling(0, 2)
b.step(5)
limits = [x.split() for x in calls("attr")]
for kernel in ("k_deliver_part", "k_deliver_words", "k_deliver_cluster", "k_deliver_stream", "k_adjoint", "k_step", "k_batch"):
    assert any(kernel in x[1] for x in limits), kernel
assert {x[2] for x in limits} == {"232448"}, {(x[1], x[2]) for x in limits if x[2] != "232448"}
""")


def test_ring_copies_without_device_memory(run):
    """Reading, saving and loading the ring where the device has no room for
    its staging copy."""
    run("""
net = pkg.Microcircuit(workload.microcircuit(0.02), stream=Stream(), raster_capacity=1 << 16, n_part=7)
most, n = net.info()["max_part_neurons"], net.n
lo = np.arange(8) * n // 7
ring = words(7 * 64 * most).view(np.int32).reshape(7, 64, most)
want = np.random.default_rng(1).integers(-9, 9, (64, n)).astype(np.int32)
for c in range(7):
    ring[c, :, :lo[c + 1] - lo[c]] = want[:, lo[c]:lo[c + 1]]
rt.fake_alloc_limit(1 << 12)
assert (net.ring() == want).all()
saved = net.save_state()
ring[:] = -1
net.load_state(saved)
assert (net.ring() == want).all() and (ring[:, :, most - 1][np.diff(lo) < most] == 0).all()
""")


def test_batches_that_have_no_room_side_by_side(run):
    """The batch kernel takes a batch whose decoded rows do not fit."""
    run("""
cfgs = [workload.microcircuit(0.13)]
kw = dict(stream=Stream(), raster_capacity=1 << 16)
assert pkg.MicrocircuitBatch(cfgs, **kw).info(0)["blocks"] < 152
rt.fake_clear()
rt.fake_alloc_limit(4 * workload.n_neurons(cfgs[0]) * 60)       # less than the table of the runs of 63 partitions
b = pkg.MicrocircuitBatch(cfgs, **kw)
assert b.info(0)["blocks"] == 152
b.step(3)
assert any("k_batch" in x for x in calls("launch"))
""")


def test_arrays_of_a_large_read_are_given_back(run):
    """What a read sorts in is kept for the next one, up to 100 MB."""
    run("""
for make in (lambda: pkg.Microcircuit(workload.microcircuit(0.02), stream=Stream(), raster_capacity=6 << 20, n_part=1),
             lambda: pkg.MicrocircuitBatch([workload.microcircuit(0.02)] * 2, stream=Stream(), raster_capacity=6 << 20)):
    h = make()
    many = [np.empty(5 << 20, np.uint32) for _ in range(2)]
    read = (lambda: h.read_spikes_into(*many)) if isinstance(h, pkg.Microcircuit) else (lambda: h.read_spikes_into(0, *many))
    h.step(3)
    read()
    for n, kept in ((2 << 20, True), (5 << 20, False), (1 << 20, True)):
        h.step(3)
        rt.fake_raster_count()[0] = n
        assert read() == n
        assert bool(rt.fake_alloc(4 * n, 1)) == kept and bool(rt.fake_alloc(16 * n, 0)) == kept, n
    h.close()
""")


def test_first_gradients_decode_rows_only_where_they_can_fit(run):
    """The rows are cut and decoded for the adjoint's partitions only where the
    partition-local form is possible, and it is done without where there is no
    room for that."""
    run("""
rng = np.random.default_rng(2)


def backward(per_row, limit=1 << 40):
    cfg = workload.microcircuit(0.12)
    n = workload.n_neurons(cfg)
    rp = np.arange(n + 1) * per_row
    targets = np.sort(rng.integers(0, n, (n, per_row)), 1).astype(np.uint32).ravel()
    net = pkg.Microcircuit(cfg, stream=Stream(), raster_capacity=1 << 16,
                           rows={"row_ptr": rp, "words": targets | np.uint32(1 << 19),
                                 "wtab": np.ones((8, 8, 128), np.int32)})
    assert net.info()["n_part"] > -(-n // 512)
    net.grad_forward(4, 2)
    rt.fake_clear()
    rt.fake_alloc_limit(limit)
    net.grad_backward(np.ones(8))
    rt.fake_alloc_limit(1 << 40)
    decoded = [x for x in calls("malloc") if int(x.split()[-1]) == 4 * (n * per_row + 4)]
    kernel = [x.split()[1] for x in calls("launch") if "k_adjoint" in x and "fold" not in x][-1]
    net.close()
    return len(decoded), "k_adjoint_part" in kernel


assert backward(300) == (1, True)
assert backward(1000) == (0, False)             # 246 KB of rows for every CTA
assert backward(300, 8 << 20) == (1, False)     # tried, no room for 11 MB
""")
