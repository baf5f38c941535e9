"""GPU tests: which launches bucket_kernel starts, and its split of large events.
An event is bucketed by a cluster of eight blocks, a step a block, so the
largest one decides where the host knows it; where the offsets are the
device's, larger ones are split among several clusters.  Seen by the kernels
launched (three with it); results against the oracle on both sides of each
line."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches
from tests.test_gpu_small_launch import _events, _run

pytestmark = pytest.mark.gpu

MOST = 131008  # digis of the largest event that a cluster takes


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert torch.cuda.get_device_properties(0).multi_processor_count // 8 == 19
    return torch


# modules, sizes of the events, kernels of the host entries, kernels of the device entry
CASES = [(64, [MOST], 3, 3), (64, [MOST + 1], 5, 5), (64, [1, MOST, 3], 3, 3), (64, [3, MOST - 5, 2], 3, 3),
         (64, [5, MOST + 1], 5, 3), (64, [100000] * 4, 3, 3), (64, [400000, 30000, 30000, 30000], 5, 3),
         (64, [0, 7, 300000] + [1000] * 12, 5, 3), (64, [131000] * 4, 3, 3), (64, [2000] * 19, 3, 3),
         (64, [2000] * 20, 5, 5), (64, [7] * 9 + [MOST * 2, 13, MOST * 2 + 1] + [0] * 3, 5, 3),
         (64, [600001, 3, 0, 70000, 1, 5], 6, 3), (64, [1] * 8 + [1000003], 6, 3), (64, [12, 262005], 5, 3),
         (64, [12, 262006], 5, 5), (1, [40000, 20000], 3, 3), (2047, [9, 270001, 11], 5, 3), (300, [200003] * 5, 6, 5)]


@pytest.mark.parametrize("M,sizes,host,device", CASES)
def test_routes_match_the_oracle(torch_cuda, M, sizes, host, device):
    words, mods, offs = _events(sizes, M, len(sizes) + sizes[0])
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        ev = ctx.enqueue_batch(words, mods, offs, flags=hp.HP_WANT_LABELS)
        assert ev.wait(60) == hp.HP_OK
        assert_batch_matches(ev.fetch(), ref, offs)
        ev.release()
        k = ctx.stats()["kernel_launches"]
        assert k == host
        for shift in (0, 1):  # inputs aligned to 16 bytes, and not
            got = _run(torch_cuda, ctx, words, mods, offs, shift).to_result(len(words))
            assert_batch_matches(got, ref, offs)
        assert ctx.stats()["kernel_launches"] - k == 2 * device


def test_invalid_modules_and_offsets_with_split_events(torch_cuda):
    M, sizes = 64, [20, 400000, 30000, 0, 150000]
    words, mods, offs = _events(sizes, M, 3)
    gain, ped = synth.calibration(M, 6)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        for at in (25, 200000, 399999):  # in each part of the event
            broken = mods.copy()
            broken[at] = M
            got = _run(torch_cuda, ctx, words, broken, offs).to_result(len(words))
            assert got.event_status.tolist() == [hp.HP_OK, hp.HP_EBADDIGI] + [hp.HP_OK] * 3
            assert_batch_matches(got, oracle.reconstruct_batch(words, broken, offs, M, gain, ped), offs)
        N = len(words)
        for k, v in ((0, 1), (5, N - 1), (1, N + 5), (2, 0), (3, N), (2, N + 1), (1, 1 << 40)):
            o = offs.copy()
            o[k] = v
            got = _run(torch_cuda, ctx, words, mods, o).to_result(N)
            if k == 3 and v == N:  # 0, 20, 400020, N, 430020: runs backwards
                assert o[3] > o[4]
            assert np.all(got.event_status == hp.HP_EINVAL) and np.all(got.cluster_offsets == 0), (k, v)
        assert_batch_matches(_run(torch_cuda, ctx, words, mods, offs).to_result(N), ref, offs)
