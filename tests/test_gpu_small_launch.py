"""GPU tests of the small launches' kernels (bucket_kernel: a cluster of
blocks an event; finish_kernel: every block scans the items), against the
oracle: event sizes around a thread's group, a block's step and the lines to
the other kernels, empty events, unaligned event starts and inputs, module
counts around four a thread and the largest, invalid modules, offsets that do
not fit, and outputs too small for the clusters."""
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


def _events(sizes, M, seed):
    """Unique pixels in random order, modules uneven (about one digi in four on module 0)."""
    rng = np.random.default_rng(seed)
    ws, ms = [], []
    for n in sizes:
        key = rng.choice(M * 66560, size=n, replace=False) if n else np.empty(0, np.int64)
        key = np.where((rng.random(n) < 0.25) & (n < 66560), key % 66560, key)
        key = rng.permutation(np.unique(key))
        extra = np.setdiff1d(np.arange(min(M * 66560, 2 * n + 2)), key)[:n - len(key)]
        key = np.concatenate([key, extra])
        m, lin = key // 66560, key % 66560
        ws.append(synth.pack(lin // 416, lin % 416, rng.integers(1, 256, n)))
        ms.append(m.astype(np.uint16))
    return np.concatenate(ws), np.concatenate(ms), np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)


def _run(torch, ctx, words, mods, offs, shift=0, capacity=None):
    dev = torch.device("cuda:0")
    E, N = len(offs) - 1, len(words)
    d_w = torch.zeros(N + 8, dtype=torch.int32, device=dev)
    d_m = torch.zeros(N + 8, dtype=torch.int16, device=dev)
    d_w[shift:shift + N] = torch.from_numpy(words.view(np.int32)).to(dev)
    d_m[shift:shift + N] = torch.from_numpy(mods.view(np.int16)).to(dev)
    d_o = torch.from_numpy(offs.view(np.int64)).to(dev)
    out = hp.DeviceOutputs(E, N, dev, capacity=capacity)
    ctx.reconstruct_device(E, N, d_o.data_ptr(), d_w[shift:].data_ptr(), d_m[shift:].data_ptr(), out,
                           torch.cuda.current_stream(dev).cuda_stream)
    torch.cuda.synchronize(dev)
    return out


CASES = [(64, [1]), (64, [7]), (64, [8]), (64, [9]), (64, [0]), (1, [5000]), (3, [16383]), (4, [16384]), (5, [16385]),
         (64, [131071]), (64, [131072]), (64, [131073]), (64, [300000]), (257, [4097]), (2047, [70001]),
         (2048, [70000]), (2049, [70000]), (4096, [9000]), (64, [0, 13, 0, 0, 4099, 8, 200001, 1]),
         (300, [777] * 9 + [0]), (1856, [3000] * 9)]


@pytest.mark.parametrize("M,sizes", CASES)
def test_sizes_around_the_lines(torch_cuda, M, sizes):
    words, mods, offs = _events(sizes, M, M + len(sizes))
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        for shift in (0, 1):
            got = _run(torch_cuda, ctx, words, mods, offs, shift).to_result(len(words))
            assert_batch_matches(got, ref, offs)
        ev = ctx.enqueue_batch(words, mods, offs, flags=hp.HP_LABELS_U16)
        assert ev.wait(60) == hp.HP_OK
        g16 = ev.fetch()
        ev.release()
        assert_batch_matches(g16, ref, offs)
        assert np.array_equal(g16.labels_from_compact(offs, mods), ref.label)


def test_invalid_modules_and_offsets(torch_cuda):
    M = 64
    gain, ped = synth.calibration(M, 6)
    for sizes, bad in (([5000], 0), ([1000, 20000, 3000], 1)):
        words, mods, offs = _events(sizes, M, 3)
        broken = mods.copy()
        broken[int(offs[bad]) + sizes[bad] // 2] = M
        expect = [hp.HP_EBADDIGI if e == bad else hp.HP_OK for e in range(len(sizes))]
        with hp.Context(M, gain, ped) as ctx:
            got = _run(torch_cuda, ctx, words, broken, offs).to_result(len(words))
            assert got.event_status.tolist() == expect
            ref = oracle.reconstruct_batch(words, broken, offs, M, gain, ped)
            assert_batch_matches(got, ref, offs)
            for k, v in ((0, 1), (len(sizes), len(words) - 1), (1, len(words) + 5)):
                o = offs.copy()
                o[k] = v
                got = _run(torch_cuda, ctx, words, mods, o).to_result(len(words))
                assert np.all(got.event_status == hp.HP_EINVAL) and np.all(got.cluster_offsets == 0)
            ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)  # and the next call is exact
            assert_batch_matches(_run(torch_cuda, ctx, words, mods, offs).to_result(len(words)), ref, offs)


def test_too_small_outputs(torch_cuda):
    words, mods, offs = _events([4000, 3000], 64, 9)
    gain, ped = synth.calibration(64, 7)
    ref = oracle.reconstruct_batch(words, mods, offs, 64, gain, ped)
    with hp.Context(64, gain, ped) as ctx:
        for cap in (ref.n_clusters - 1, 1):
            out = _run(torch_cuda, ctx, words, mods, offs, capacity=cap)
            assert out.event_status.tolist() == [hp.HP_ECAPACITY] * 2
            assert out.id[:cap].cpu().numpy().tolist() == ref.id[:cap].tolist()
        out = _run(torch_cuda, ctx, words, mods, offs, capacity=ref.n_clusters)
        assert out.event_status.tolist() == [hp.HP_OK] * 2
