"""GPU tests of the clustering kernel with three groups of 160 threads a block,
which takes launches of many small or of large items: sizes around its own
lines (packs of 640 digis, 1,280 held by a group, items past 1,800 by the whole
block, 3,840 held by it), clusters that need the 64-bit moments in each tier,
and invalid and duplicated digis in each, against the oracle.  The launches'
shape is worked out with the library's own rule, so that a moved line shows."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches
from tests.test_launch_sizes import host_program

pytestmark = pytest.mark.gpu

ROWS, COLS = 160, 416


def _random(rng, n, lo=1):
    lin = rng.choice(ROWS * COLS, size=n, replace=False)
    return synth.pack(lin // COLS, lin % COLS, rng.integers(lo, 256, n)).astype(np.uint32)


def _block(h, w):
    r, c = np.meshgrid(np.arange(h) + 20, np.arange(w) + 100, indexing="ij")
    return synth.pack(r.ravel(), c.ravel(), np.full(h * w, 250)).astype(np.uint32)


def _check(tmp_path, events, gain, expect=None):
    """events: lists of the modules' words."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(4)
    E, M = len(events), len(events[0])
    ws, ms, offs = [], [], [0]
    for ev in events:
        w, m = np.concatenate(ev), np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(ev)])
        perm = rng.permutation(len(w))
        ws.append(w[perm])
        ms.append(m[perm])
        offs.append(offs[-1] + len(w))
    words, mods, offs = np.concatenate(ws), np.concatenate(ms), np.asarray(offs, np.uint64)
    N, items = len(words), E * M
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    grid = min(items if N >= 64 * items else (items + 3) // 4, 2 * sms)
    shape = host_program(tmp_path, f"""hp::Tuning t; hp::RunShape s = hp::run_shape(t, {items}, {N}, {grid});
        printf("%u %u %u", s.threads, s.groups, hp::large_digis({ROWS}, {COLS}, t.tile_slots, s));""")
    assert shape == "480 3 1800"
    gain, ped = np.full(M, gain, np.int32), np.full(M, 50, np.int32)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        assert ctx.get_tuning(E, N)["blocks_per_sm"] == 2 and ctx.get_tuning(E, N)["tile_slots"] == 4096
        for flags in (hp.HP_WANT_LABELS, hp.HP_LABELS_U16):
            ev = ctx.enqueue_batch(words, mods, offs, flags=flags)
            ev.wait(60)
            got = ev.fetch()
            ev.release()
            assert expect is None or got.event_status.tolist() == expect
            assert_batch_matches(got, ref, offs)
            if flags == hp.HP_LABELS_U16 and not ref.event_status.any():
                assert np.array_equal(got.labels_from_compact(offs, mods), ref.label)


SIZES = [639, 640, 641, 767, 768, 769, 1279, 1280, 1281, 1799, 1800, 1801, 3839, 3840, 3841, 4500, 0, 1]


@pytest.mark.parametrize("per", [70, 90])  # packs of one and of several of the other items
def test_sizes_around_the_lines(tmp_path, per):
    rng = np.random.default_rng(per)
    sizes = np.concatenate([SIZES, rng.integers(per - 20, per + 20, 900)])
    _check(tmp_path, [[_random(rng, n) for n in rng.permutation(sizes)]], 70)


def test_large_items(tmp_path):
    """Items of 640 digis and more on average."""
    rng = np.random.default_rng(2)
    _check(tmp_path, [[_random(rng, n) for n in rng.permutation(np.concatenate([SIZES, rng.integers(700, 1000, 640)]))]],
           70)


def test_heavy_clusters(tmp_path):
    assert 15 * 16 * 250 * 126 > 0x7FFFFFFF // 512
    rng = np.random.default_rng(3)
    dense = [_block(15, 16), _block(25, 25), _block(30, 40), _block(40, 44), _block(50, 60), _block(60, 75)]
    _check(tmp_path, [dense + [_random(rng, int(n)) for n in rng.integers(60, 100, 700)]], 126)


def test_invalid_and_duplicated_digis(tmp_path):
    rng = np.random.default_rng(5)
    ok = [_random(rng, n, 20) for n in (100, 620, 1000, 1500, 2500)] + [_random(rng, 70, 20) for _ in range(145)]
    events, expect = [ok], [hp.HP_OK]
    for k in range(5):
        for bad in ("dup", "dropped", "adc"):
            ev = [x.copy() for x in ok]
            w = ev[k][0]
            if bad == "adc":
                ev[k][0] = w & np.uint32(0x1FFFF)
            else:
                ev[k] = np.append(ev[k], w if bad == "dup" else (w & np.uint32(0x1FFFF)) | np.uint32(1 << 17))
            events.append(ev)
            expect.append(hp.HP_EBADDIGI if bad == "adc" else hp.HP_EDUP)
    _check(tmp_path, events + [ok], 70, expect + [hp.HP_OK])
