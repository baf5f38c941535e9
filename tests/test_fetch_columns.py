"""The six cluster columns of a fetched product (CPU case of the library, and
plain arrays): right types and values, writable, in place or copied; one memory
view for all of them where they lie at one stride, whatever their length."""
import numpy as np
import pytest

from paper_2004_04334_gb300 import hp, synth

TYPES = (np.uint32, np.int32, np.int32, np.int32, np.float32, np.float32)


def _check(base, ptrs, n, offs):
    cols = hp._columns(ptrs, n, copy=False)
    copies = hp._columns(ptrs, n)
    for k, (c, d, t, o) in enumerate(zip(cols, copies, TYPES, offs)):
        assert c.dtype == d.dtype == t and c.shape == d.shape == (n,) and c.flags.writeable and d.flags.writeable
        want = base[o:o + n].view(t)
        assert np.array_equal(c, want) and np.array_equal(d, want)
        if n:
            assert c.ctypes.data == ptrs[k]
            base[o] += 1
            assert c[0] == base[o:o + 1].view(t)[0] and d[0] != c[0]


@pytest.mark.parametrize("n", [0, 1, 5, 64])
@pytest.mark.parametrize("starts", [[64 * k for k in range(6)], [70 * k + 3 for k in range(6)],
                                    [0, 64, 128, 192, 256, 330], [330, 256, 192, 128, 64, 0]])
def test_columns(n, starts):
    base = np.arange(1000, 1500, dtype=np.int32)
    _check(base, tuple(base.ctypes.data + 4 * s for s in starts), n, starts)


def test_no_columns():
    for ptrs in ((None,) * 6, (4096,) * 6):
        assert [(c.dtype, c.shape) for c in hp._columns(ptrs, 0)] == [(np.dtype(t), (0,)) for t in TYPES]


def test_a_fetch_makes_one_view_of_its_columns(monkeypatch):
    w = synth.workload("tiny", n_events=2)
    monkeypatch.setenv("HP_FORCE_CPU", "1")
    views = []
    make = hp._memory
    monkeypatch.setattr(hp, "_memory", lambda *a: views.append(a) or make(*a))
    with hp.Context(w.n_modules, w.gain, w.pedestal) as ctx:
        ev = ctx.enqueue_batch(w.words, w.modules, w.offsets)
        ev.wait(60)
        got = ev.fetch(copy=False)
        assert got.n_clusters > 0 and len(views) == 3  # the event offsets, the statuses, the columns
        ev.release()
