"""GPU tests of the clustering of few items (no more than blocks): a block
clusters its own item, whole or by one of its groups as the item's size has it.
Sizes around that line, numbers of items around the blocks', against the
oracle; and a time: items of 2,000 digis, some of them past the line, take no
longer than larger ones."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches

pytestmark = pytest.mark.gpu

LINE = 1280  # five digis a thread of a group of 256


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _event(sizes, seed):
    rng = np.random.default_rng(seed)
    lin = [rng.choice(160 * 416, size=n, replace=False) for n in sizes]
    words = np.concatenate([synth.pack(x // 416, x % 416, rng.integers(1, 256, len(x))) for x in lin]).astype(np.uint32)
    mods = np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(lin)])
    perm = rng.permutation(len(words))
    return words[perm], mods[perm]


EDGES = [LINE - 1, LINE, LINE + 1, 2047, 2048, 2049, 4095, 4096, 8191, 8193, 20000, 0, 1, 767, 769]


@pytest.mark.parametrize("sizes", [EDGES, EDGES + [LINE + 1] * 137, EDGES + [LINE - 1, LINE + 1] * 69,
                                   [900, LINE + 1] * 152, [900, LINE + 1] * 152 + [5]])
def test_few_items_match_the_oracle(torch_cuda, sizes):
    """15, 152, 153, 304 and 305 items: one block an SM has 152, two have 304."""
    M = len(sizes)
    words, mods = _event(sizes, M)
    offs = np.array([0, len(words)], np.uint64)
    gain, ped = np.full(M, 70, np.int32), np.full(M, 50, np.int32)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        settings = [t for t in ctx.tuning_candidates() if t["label_store"] == hp.HP_STORE_BITMAP and t["warp_max"] == 64
                    and t["ticket_items"] in (4, 16)]
        for t in [ctx.get_tuning(1, len(words))] + settings:
            ctx.set_tuning(1, len(words), t)
            for flags in (hp.HP_WANT_LABELS, hp.HP_LABELS_U16):
                ev = ctx.enqueue_event(words, mods, flags=flags)
                assert ev.wait(60) == hp.HP_OK
                got = ev.fetch()
                ev.release()
                assert_batch_matches(got, ref, offs)
                if flags == hp.HP_LABELS_U16:
                    assert np.array_equal(got.labels_from_compact(offs, mods), ref.label), t


def test_items_around_the_line_take_no_longer_than_larger_ones(torch_cuda):
    torch = torch_cuda
    dev = torch.device("cuda:0")
    stream = torch.cuda.current_stream(dev).cuda_stream
    M, runs = 128, []
    with hp.Context(M, *synth.calibration(M, 2004)) as ctx:
        for mean in (2000, 2600):
            noise = synth.TINY.lambda_noise
            words, mods = synth.make_event(replace(synth.TINY, n_modules=M, lambda_clusters=(mean - noise) / 6.5), mean)
            N = len(words)
            d = [torch.from_numpy(a).to(dev) for a in (np.array([0, N]), words.view(np.int32), mods.view(np.int16))]
            out = hp.DeviceOutputs(1, N, dev)
            runs.append((lambda N=N, d=d, out=out: ctx.reconstruct_device(1, N, *[x.data_ptr() for x in d], out, stream)))
        best = [1e9, 1e9]
        for _ in range(8):
            for i, run in enumerate(runs):
                for _ in range(3):
                    run()
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(20):
                    run()
                b.record()
                torch.cuda.synchronize(dev)
                best[i] = min(best[i], a.elapsed_time(b) / 20)
    assert best[0] <= 1.15 * best[1], best
