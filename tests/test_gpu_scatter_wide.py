"""GPU tests of the scatter for many modules (scatter_wide_kernel) against
the oracle: steps inside one event, steps over several events (with the keys
in the shared tables, and past them), more events than the offsets kept in
shared memory, a last step that is nearly empty, unaligned inputs, and invalid
modules."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches

pytestmark = pytest.mark.gpu

STEP = 16384  # digis a block sorts at a time


@pytest.mark.parametrize("M,sizes,bad", [
    (257, [2600000], False),
    (1856, [152 * STEP + 1, 70001, 13], False),
    (300, [5, 0, 900000, 3, 1600000] + [9], True),
    (4096, [900000, 850000, 800000], False),
    (300, [0, 7] * 258 + [2500000, 3000000, 3100000], False),
])
def test_matches_the_oracle(M, sizes, bad):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N = int(sum(sizes))
    assert N >= 152 * STEP and N // len(sizes) >= STEP
    rng = np.random.default_rng(M)
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    ws, ms = [], []
    for n in sizes:  # every pixel of the event once: an odd multiplier walks them all
        space = M * 66560
        start, stride = int(rng.integers(space)), 2 * int(rng.integers(space // 4)) + 1
        while np.gcd(stride, space) != 1:
            stride += 2
        key = (start + np.arange(n, dtype=np.int64) * stride) % space
        ms.append((key // 66560).astype(np.uint16))
        lin = key % 66560
        ws.append(synth.pack(lin // 416, lin % 416, rng.integers(1, 256, n)))
    words, mods = np.concatenate(ws), np.concatenate(ms)
    if bad:
        mods[int(offs[2]) + 100] = M  # event 2
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    assert bool(ref.event_status.any()) == bad
    dev = torch.device("cuda:0")
    with hp.Context(M, gain, ped) as ctx:
        for shift in (0, 1):
            d_w = torch.zeros(N + 8, dtype=torch.int32, device=dev)
            d_m = torch.zeros(N + 8, dtype=torch.int16, device=dev)
            d_w[shift:shift + N] = torch.from_numpy(words.view(np.int32)).to(dev)
            d_m[shift:shift + N] = torch.from_numpy(mods.view(np.int16)).to(dev)
            d_o = torch.from_numpy(offs.view(np.int64)).to(dev)
            out = hp.DeviceOutputs(len(sizes), N, dev)
            ctx.reconstruct_device(len(sizes), N, d_o.data_ptr(), d_w[shift:].data_ptr(), d_m[shift:].data_ptr(), out,
                                   torch.cuda.current_stream(dev).cuda_stream)
            torch.cuda.synchronize(dev)
            assert_batch_matches(out.to_result(N), ref, offs)
