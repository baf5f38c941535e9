"""GPU test: which launches bucket_kernel starts.  An event is bucketed by eight
blocks, so the largest one decides where the host knows it, and the launch's
digis where the offsets are the device's.  Seen by the kernels launched (three
with it); results against the oracle on both sides of each line."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches
from tests.test_gpu_small_launch import _events

pytestmark = pytest.mark.gpu

M, MOST = 64, 131008  # digis of the largest event that bucket_kernel takes

# sizes of the events, kernels of the host entries, kernels of the device entry
CASES = [([MOST], 3, 3), ([MOST + 1], 5, 5), ([1, MOST, 3], 3, 5), ([3, MOST - 5, 2], 3, 3), ([5, MOST + 1], 5, 5),
         ([100000] * 4, 3, 5), ([400000, 30000, 30000, 30000], 5, 5), ([0, 7, 300000] + [1000] * 12, 5, 5),
         ([131000] * 4, 3, 5), ([2000] * 19, 3, 3), ([2000] * 20, 5, 5)]


@pytest.mark.parametrize("sizes,host,device", CASES)
def test_the_largest_event_decides(sizes, host, device):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert torch.cuda.get_device_properties(0).multi_processor_count // 8 == 19
    words, mods, offs = _events(sizes, M, len(sizes) + sizes[0])
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    E, N = len(sizes), len(words)
    dev = torch.device("cuda:0")
    d = [torch.from_numpy(a.view(t)).to(dev) for a, t in ((offs, np.int64), (words, np.int32), (mods, np.int16))]
    out = hp.DeviceOutputs(E, N, dev)
    with hp.Context(M, gain, ped) as ctx:
        ev = ctx.enqueue_batch(words, mods, offs, flags=hp.HP_WANT_LABELS)
        assert ev.wait(60) == hp.HP_OK
        assert_batch_matches(ev.fetch(), ref, offs)
        ev.release()
        k = ctx.stats()["kernel_launches"]
        assert k == host
        ctx.reconstruct_device(E, N, *[x.data_ptr() for x in d], out, torch.cuda.current_stream(dev).cuda_stream)
        torch.cuda.synchronize(dev)
        assert_batch_matches(out.to_result(N), ref, offs)
        assert ctx.stats()["kernel_launches"] - k == device
