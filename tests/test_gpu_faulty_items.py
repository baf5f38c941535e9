"""GPU test: an item (event, module) with an invalid or a duplicated digi keeps
no cluster and gets no labels, whichever tier clusters it; the event's other
items and the other events are exact, and an output that holds their clusters
and no more is enough."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth

pytestmark = pytest.mark.gpu

M, ROWS, COLS = 5, 160, 416
SIZES = [24, 60, 300, 700, 2500]  # the packed tier under every setting, under most, and the tiers above it
KINDS = ["dup", "dropped", "adc", "row", "high"]
UNTOUCHED = 123456789


def _events():
    """Good events before, between and after the faulty ones: (words, modules, faulty module or None, status)."""
    rng = np.random.default_rng(12)
    lin = [rng.choice(ROWS * COLS, size=n, replace=False) for n in SIZES]
    ok = [synth.pack(x // COLS, x % COLS, rng.integers(60, 200, len(x))).astype(np.uint32) for x in lin]
    events = [(ok, None, hp.HP_OK)]
    for k in range(M):
        for kind in KINDS:
            ev = [x.copy() for x in ok]
            w = ev[k][0]
            if kind in ("dup", "dropped"):  # its pixel once more, above or below threshold
                ev[k] = np.append(ev[k], w if kind == "dup" else (w & np.uint32(0x1FFFF)) | np.uint32(1 << 17))
            else:
                ev[k][0] = {"adc": w & np.uint32(0x1FFFF), "row": (w & ~np.uint32(0xFF)) | np.uint32(ROWS),
                            "high": w | np.uint32(1 << 31)}[kind]
            events.append((ev, k, hp.HP_EDUP if kind in ("dup", "dropped") else hp.HP_EBADDIGI))
    events.append((ok, None, hp.HP_OK))
    out = []
    for items, k, status in events:
        m = np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(items)])
        perm = rng.permutation(len(m))
        out.append((np.concatenate(items)[perm], m[perm], k, status))
    return out


def test_a_faulty_item_keeps_nothing_in_any_tier():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    events = _events()
    gain, ped = np.full(M, 70, np.int32), np.full(M, 50, np.int32)
    # the reference: the events without their faulty items
    refs = [oracle.reconstruct_event(w[m != k] if k is not None else w, m[m != k] if k is not None else m, M, gain, ped)
            for w, m, k, _ in events]
    total = sum(r.n_clusters for r in refs)
    words, mods = (np.concatenate([e[i] for e in events]) for i in (0, 1))
    offs = np.concatenate([[0], np.cumsum([len(e[0]) for e in events])]).astype(np.uint64)
    E, N = len(events), len(words)
    dev = torch.device("cuda:0")
    d = [torch.from_numpy(a.view(t)).to(dev) for a, t in ((offs, np.int64), (words, np.int32), (mods, np.int16))]
    out = hp.DeviceOutputs(E, N, dev, capacity=total)
    stream = torch.cuda.current_stream(dev).cuda_stream
    with hp.Context(M, gain, ped) as ctx:
        for t in ctx.tuning_candidates():
            ctx.set_tuning(E, N, t)
            out.label.fill_(UNTOUCHED)
            ctx.reconstruct_device(E, N, *[x.data_ptr() for x in d], out, stream)
            torch.cuda.synchronize(dev)
            got = out.to_result(N)
            assert got.event_status.tolist() == [e[3] for e in events], t
            assert np.diff(got.cluster_offsets.astype(np.int64)).tolist() == [r.n_clusters for r in refs], t
            for f in ("module", "id", "charge", "npix"):
                assert np.array_equal(getattr(got, f), np.concatenate([getattr(r, f) for r in refs])), (f, t)
            for (w, m, k, _), r, a in zip(events, refs, offs[:-1].astype(int)):
                label = got.label[a:a + len(w)]
                bad = m == k if k is not None else np.zeros(len(m), bool)
                assert np.array_equal(label[~bad], r.label), t
                assert np.all(label[bad] == UNTOUCHED), t
