"""GPU tests of the clustering kernel's packed and run tiers against the
oracle, under one, two and three blocks per SM: module geometries around the
bitmap's word size, item sizes on both sides of every tier's line (the packed
tier's largest item and pack, the digis a group holds in registers, whole-
block items, more runs than a slice or a block holds), clusters heavy enough
for the 64-bit moments in each tier, and invalid or duplicated digis in each.
Centroids within 1e-4 pixel (the repository's tolerance), all else equal."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _check(items, gain, ped, rows=160, cols=416, expect=None):
    """items: one list of digi words per (event, module); every bitmap setting, both label forms."""
    E, M = len(items), len(items[0])
    rng = np.random.default_rng(3)
    ws, ms, offs = [], [], [0]
    for ev in items:
        w = np.concatenate(ev).astype(np.uint32)
        m = np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(ev)])
        perm = rng.permutation(len(w))
        ws.append(w[perm])
        ms.append(m[perm])
        offs.append(offs[-1] + len(w))
    words, mods, offs = np.concatenate(ws), np.concatenate(ms), np.asarray(offs, np.uint64)
    N = int(offs[-1])
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped, rows=rows, cols=cols)
    with hp.Context(M, gain, ped, rows=rows, cols=cols) as ctx:
        seen = set()
        for t in ctx.tuning_candidates():
            key = (t["blocks_per_sm"], t["warp_max"])
            if t["label_store"] != hp.HP_STORE_BITMAP or key in seen:
                continue
            seen.add(key)
            ctx.set_tuning(E, N, t)
            for flags in (hp.HP_WANT_LABELS, hp.HP_LABELS_U16):
                ev = ctx.enqueue_batch(words, mods, offs, flags=flags)
                ev.wait(120)
                got = ev.fetch()
                ev.release()
                if expect is not None:
                    assert got.event_status.tolist() == expect, t
                assert_batch_matches(got, ref, offs)
                if flags == hp.HP_LABELS_U16 and not ref.event_status.any():
                    assert np.array_equal(got.labels_from_compact(offs, mods), ref.label), t
        assert {b for b, _ in seen} == {1, 2, 3}


def _random(n, rng, rows=160, cols=416, adc=(1, 256)):
    lin = rng.choice(rows * cols, size=n, replace=False)
    return synth.pack(lin // cols, lin % cols, rng.integers(adc[0], adc[1], n))


@pytest.mark.parametrize("rows,cols", [(256, 340), (256, 1), (1, 512), (5, 31), (9, 32), (30, 33), (200, 65), (160, 416)])
def test_geometries(torch_cuda, rows, cols):
    rng = np.random.default_rng(rows * cols)
    px = rows * cols
    items = [[_random(max(1, int(f * px)), rng, rows, cols) for f in fs] for fs in ((0.02, 0.6, 1.0), (0.1, 0.3, 0.9))]
    _check(items, np.array([60, 30, 64], np.int32), np.array([0, 100, 16], np.int32), rows, cols)


def test_item_sizes_around_the_tiers_lines(torch_cuda):
    rng = np.random.default_rng(5)
    sizes = [[1, 64, 65, 255, 256, 257, 511, 512], [513, 1023, 1024, 2047, 2048, 2049, 0, 3],
             [300, 300, 300, 300, 300, 2000, 300, 256], [3100, 3300, 5000, 8193, 12000, 40000, 7, 66560]]
    items = [[_random(n, rng) for n in row] for row in sizes]
    _check(items, np.full(8, 70, np.int32), np.full(8, 50, np.int32))


def test_more_runs_than_shared_memory_holds(torch_cuda):
    """Isolated pixels (a run each): more than a slice, a block, and as many as a module has."""
    rng = np.random.default_rng(6)
    r, c = np.meshgrid(np.arange(160), np.arange(0, 416, 2), indexing="ij")
    every = synth.pack(r.ravel(), c.ravel(), np.full(r.size, 90))  # 33,280 runs, joined by rows
    lone = every[(r.ravel() % 2) == 0]                             # 16,640, none adjacent
    pick = lambda n: rng.choice(lone, size=n, replace=False)  # noqa: E731
    _check([[pick(2100), pick(2200), pick(3000)], [pick(4000), every, lone], [pick(11000), pick(600), pick(100)]],
           np.full(3, 70, np.int32), np.full(3, 0, np.int32))


def test_heavy_clusters(torch_cuda):
    """Dense blocks whose moments overflow 32 bits, in the packed tier, a group's and a whole block's run tier."""
    def block(h, w):
        rr, cc = np.meshgrid(np.arange(h) + 60, np.arange(w) + 100, indexing="ij")
        return synth.pack(rr.ravel(), cc.ravel(), np.full(h * w, 250))
    items = [[block(15, 16), block(30, 60), block(50, 60)], [block(90, 100), block(3, 3), block(30, 40)]]
    gain = np.full(3, 126, np.int32)
    assert 240 * 250 * 126 > 0x7FFFFFFF // 512
    _check(items, gain, np.zeros(3, np.int32))


def test_invalid_and_duplicated_digis(torch_cuda):
    rng = np.random.default_rng(8)
    sizes = [100, 1500, 3000, 6000]
    ok = [_random(n, rng, adc=(20, 200)) for n in sizes]
    items, expect = [ok], [hp.HP_OK]
    for k in range(4):
        for bad in ("dup", "dropped", "adc", "row", "high"):
            ev = [x.copy() for x in ok]
            if bad == "dup":
                ev[k] = np.append(ev[k], ev[k][0])
            elif bad == "dropped":  # the pixel again, below threshold
                ev[k] = np.append(ev[k], (ev[k][0] & 0x1FFFF) | (1 << 17))
            else:
                ev[k][0] = {"adc": ev[k][0] & 0x1FFFF, "row": (ev[k][0] & ~np.uint32(0xFF)) | 160,
                            "high": ev[k][0] | (1 << 31)}[bad]
            items.append(ev)
            expect.append(hp.HP_EDUP if bad in ("dup", "dropped") else hp.HP_EBADDIGI)
    items.append(ok)
    expect.append(hp.HP_OK)
    _check(items, np.full(4, 70, np.int32), np.full(4, 50, np.int32), expect=expect)


@pytest.mark.parametrize("threads", [480, 512, 1024])
def test_items_a_whole_block_holds_in_registers(torch_cuda, threads):
    """At and past eight digis a thread of a block, scattered and in one cluster that needs the 64-bit moments."""
    rng = np.random.default_rng(threads)
    line = 8 * threads
    dense = synth.pack(*(x.ravel()[:line] for x in np.meshgrid(np.arange(120) + 20, np.arange(100) + 200, indexing="ij")),
                       np.full(line, 250))
    items = [[_random(line - 1, rng), _random(line, rng), _random(line + 1, rng)], [dense, dense[:line - 1], _random(9, rng)]]
    gain = np.full(3, 126, np.int32)
    assert line * 250 * 126 * 200 > 0x7FFFFFFF
    _check(items, gain, np.zeros(3, np.int32))
