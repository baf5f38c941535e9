"""GPU tests of the histogram and the scatter over ranges of few keys
(hist_kernel, scatter_few) against the oracle: steps inside one event and over
several, full and nearly empty steps, one key and the most keys a range may
have, unaligned inputs, and invalid modules in whole groups of digis and in the
last one."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches

pytestmark = pytest.mark.gpu

KEYS = 256  # most (event, module) pairs of a range


@pytest.mark.parametrize("M,sizes,bad", [
    (64, [8191, 8192, 8193, 0, 1, 4096, 7] * 4, []),                    # half a step a block
    (64, [1700001, 3300000, 5], []),                                    # three steps a block
    (256, [4096] * 24, [4096 * 3 + 8, 4096 * 24 - 1]),                  # one event a block, 256 keys
    (1, [16] * KEYS, []),                                               # one block, an event a key
    (3, [9000] * 10 + [0] * 20 + [11] * 40, [8, 17, 9000 * 4 + 8999]),  # events end inside a step
    (1, [60000, 4, 3000] * 7, [60004]),                                 # one module
])
def test_matches_the_oracle(M, sizes, bad):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N = int(sum(sizes))
    assert N > 1 << 21 or len(sizes) * 8 > 152  # (else the digis are bucketed by another kernel)
    rng = np.random.default_rng(M + len(sizes))
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    ws, ms = [], []
    for n in sizes:  # every pixel of the event at most once: a multiplier coprime to their number walks them
        space = M * 66560
        start, stride = int(rng.integers(space)), int(rng.integers(space)) | 1
        while np.gcd(stride, space) != 1:
            stride += 2
        key = (start + np.arange(n, dtype=np.int64) * stride) % space
        ms.append((key // 66560).astype(np.uint16))
        lin = key % 66560
        ws.append(synth.pack(lin // 416, lin % 416, rng.integers(1, 256, n)))
    words, mods = np.concatenate(ws), np.concatenate(ms)
    for i, k in enumerate(bad):
        mods[k] = (M, 65535)[i % 2]
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    assert bool(ref.event_status.any()) == bool(bad)
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
