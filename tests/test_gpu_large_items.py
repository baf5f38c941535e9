"""GPU tests of the items that whole blocks take from a list (past what a
group's share of a block holds): none to more of them than there are SMs, by
one and two blocks an SM, against the oracle."""
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


def _event(sizes, seed):
    rng = np.random.default_rng(seed)
    lin = [rng.choice(160 * 416, size=n, replace=False) for n in sizes]
    words = np.concatenate([synth.pack(x // 416, x % 416, rng.integers(1, 256, len(x))) for x in lin]).astype(np.uint32)
    mods = np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(lin)])
    perm = rng.permutation(len(words))
    return words[perm], mods[perm]


@pytest.mark.parametrize("large", [0, 1, 5, 151, 152, 153, 310])
def test_lists_around_the_number_of_sms(torch_cuda, large):
    assert torch_cuda.cuda.get_device_properties(0).multi_processor_count == 152
    M = 900
    sizes = np.full(M, 150)
    sizes[np.random.default_rng(large).choice(M, large, replace=False)] = 2700
    words, mods = _event(sizes, large)
    offs = np.array([0, len(words)], np.uint64)
    gain, ped = np.full(M, 70, np.int32), np.full(M, 50, np.int32)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
    with hp.Context(M, gain, ped) as ctx:
        for t in [t for t in ctx.tuning_candidates() if t["label_store"] == hp.HP_STORE_BITMAP and
                  t["blocks_per_sm"] < 3 and t["warp_max"] == 64 and t["ticket_items"] == 16]:
            ctx.set_tuning(1, len(words), t)
            for flags in (hp.HP_WANT_LABELS, hp.HP_LABELS_U16):
                ev = ctx.enqueue_event(words, mods, flags=flags)
                assert ev.wait(60) == hp.HP_OK
                assert_batch_matches(ev.fetch(), ref, offs)
                ev.release()
