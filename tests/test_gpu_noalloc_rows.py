"""snn_step_noalloc on rows that differ from what the connection probabilities
let it expect, and on steps with more spikes than it lists at once, against
snn_step: the same spikes, state, ring buffers and counters, bit for bit."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1909_08665_gb300 as pkg  # noqa: E402


def _rows(n, kind, rng):
    """Row lengths, then targets: spread evenly, crowded into a narrow band
    that moves with the source, or one target repeated (an empty row for
    every third source)."""
    ln = rng.integers(0, min(n, 700) + 1, n)
    ln[::3] = 0
    if kind == "long":              # one row longer than a message word can say
        ln[:] = 3
        ln[0] = 1 << 22
    at = np.repeat(np.arange(n), ln)
    if kind == "even":
        tgt = rng.integers(0, n, at.size)
    elif kind == "band":
        tgt = (at * 7 + rng.integers(0, 1 + n // 50, at.size)) % n
    else:
        tgt = (at * 13) % n
        tgt[:ln[0]] = rng.integers(0, n, ln[0])
    order = np.lexsort((tgt, at))
    words = pkg.encode_words(tgt[order], rng.integers(1, 64, at.size), rng.integers(0, 128, at.size))
    return {"row_ptr": np.concatenate([[0], np.cumsum(ln)]).astype(np.uint64), "words": words,
            "wtab": rng.integers(-20000, 30000, 8 * 8 * 128).astype(np.int32)}


@pytest.mark.parametrize("scale,kind,n_above", [
    (0.0005, "even", 20),           # 38 neurons: one partition
    (0.0213, "band", 900),          # more than one list of spikes in the first step
    (0.1, "even", 3000), (0.1, "repeat", 200),
    (0.6, "band", 5000),            # the wide kernel
    (0.01, "long", 400),
])
def test_noalloc_any_rows(scale, kind, n_above):
    cfg = workload.microcircuit(scale)
    n = int(sum(cfg["pop_sizes"]))
    rng = np.random.default_rng(17)
    rows = _rows(n, kind, rng)
    u0 = workload.transient_membrane(cfg, seed=3, n_above=n_above)
    stream = torch.cuda.current_stream()
    ref = pkg.Microcircuit(cfg, u0=u0, rows=rows, stream=stream)
    cap = 1 << 20
    d = {"row_ptr": rows["row_ptr"].view(np.int64), "words": rows["words"].view(np.int32),
         "wtab": rows["wtab"], "u": u0, "i_syn": np.zeros(n, np.float32), "refr": np.zeros(n, np.int32),
         "ring": np.zeros(64 * n, np.int32), "ras_step": np.zeros(cap, np.int32),
         "ras_id": np.zeros(cap, np.int32), "ras_n": np.zeros(1, np.int32),
         "counters": np.zeros(2, np.int64), "status": np.zeros(1, np.int32)}
    d = {k: torch.from_numpy(v.copy()).cuda() for k, v in d.items()}
    io = pkg.SnnNoallocIO(ras_cap=cap, **{k: v.data_ptr() for k, v in d.items()})
    t0 = 0
    for steps in (1, 7, 150):
        pkg.step_noalloc(cfg, cfg["seed"], io, t0, steps, stream)
        ref.step(steps)
        torch.cuda.synchronize()
        assert int(d["status"].item()) == 0
        g_st, g_id = ref.read_spikes()
        m = int(d["ras_n"].item())
        st, ids = d["ras_step"][:m].cpu().numpy(), d["ras_id"][:m].cpu().numpy()
        order = np.lexsort((ids, st))
        np.testing.assert_array_equal(st[order], g_st)
        np.testing.assert_array_equal(ids[order], g_id)
        assert t0 > 0 or m >= min(n_above, n) // 2
        d["ras_n"].zero_()
        for key, want in zip(("u", "i_syn", "refr"), ref.state()):
            np.testing.assert_array_equal(d[key].cpu().numpy().view(np.uint32), want.view(np.uint32))
        np.testing.assert_array_equal(d["ring"].cpu().numpy().reshape(64, n), ref.ring())
        c = ref.counters()
        assert [int(v) for v in d["counters"].cpu()] == [c["spikes"], c["events"]]
        t0 += steps
