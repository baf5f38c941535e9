"""GPU test: which launches finish_kernel ends.  With outputs in host memory up
to 2^19 digis, with outputs kept on the device more.  Seen by the kernels
launched (five with it, of more events than bucket_kernel takes); results
against the oracle on both sides of the line."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches
from tests.test_gpu_small_launch import _events

pytestmark = pytest.mark.gpu

M = 16


@pytest.mark.parametrize("extra,host", [(0, 5), (1, 6)])
def test_where_the_outputs_are_decides(extra, host):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sizes = [16384] * 31 + [16384 + extra]
    words, mods, offs = _events(sizes, M, extra)
    gain, ped = synth.calibration(M, 5)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        seen = 0
        for flags, kernels in ((hp.HP_WANT_LABELS, host), (hp.HP_LABELS_U16, host), (hp.HP_KEEP_ON_DEVICE, 5)):
            ev = ctx.enqueue_batch(words, mods, offs, flags=flags)
            assert ev.wait(60) == hp.HP_OK
            now = ctx.stats()["kernel_launches"]
            assert now - seen == kernels, flags
            if flags == hp.HP_KEEP_ON_DEVICE:
                tr = ev.transfer()
                assert tr.wait(60) == hp.HP_OK
                got = tr.fetch()
                tr.release()
                now = ctx.stats()["kernel_launches"]
            else:
                got = ev.fetch()
            ev.release()
            seen = now
            assert_batch_matches(got, ref, offs)
