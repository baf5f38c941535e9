"""GPU test: contexts for modules of different sizes live side by side.  A
kernel's limit of dynamic shared memory belongs to the process; creating a
context must not take it below what another one's launches need."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import hp, synth
from tests.gpu_util import assert_batch_matches

pytestmark = pytest.mark.gpu


def _input(M, rows, cols, per, seed):
    rng = np.random.default_rng(seed)
    lin = np.concatenate([rng.choice(rows * cols, size=per, replace=False) for _ in range(M)])
    words = synth.pack(lin // cols, lin % cols, rng.integers(20, 256, len(lin))).astype(np.uint32)
    return words, np.repeat(np.arange(M, dtype=np.uint16), per)


# the other context's modules: larger ones, whose clustering blocks need less
# memory than the first's (smaller slices), and smaller ones
@pytest.mark.parametrize("rows,cols", [(200, 400), (80, 52)])
def test_a_context_for_other_modules_leaves_the_first_its_shared_memory(rows, cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shapes = [(700, 100), (8, 3000), (8, 400)]  # (modules, digis each): clustering blocks of each shape
    for M, per in shapes:
        gain, ped = np.full(M, 70, np.int32), np.full(M, 50, np.int32)
        words, mods = _input(M, 160, 416, per, M + per)
        offs = np.array([0, len(words)], np.uint64)
        ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped)
        w2, m2 = _input(M, rows, cols, min(per, rows * cols // 2), 1)
        offs2 = np.array([0, len(w2)], np.uint64)
        ref2 = oracle.reconstruct_batch(w2, m2, offs2, M, gain, ped, rows=rows, cols=cols)

        def check(ctx, w, m, o, r):
            ev = ctx.enqueue_batch(w, m, o, flags=hp.HP_WANT_LABELS)
            assert ev.wait(60) == hp.HP_OK
            got = ev.fetch()
            ev.release()
            assert_batch_matches(got, r, o)

        with hp.Context(M, gain, ped) as first:
            settings = [first.get_tuning(1, len(words))] + [t for t in first.tuning_candidates()
                                                            if t["ticket_items"] == 16 and t["item_threads"] == 512]
            with hp.Context(M, gain, ped, rows=rows, cols=cols) as other:
                for t in settings:
                    first.set_tuning(1, len(words), t)
                    check(first, words, mods, offs, ref)
                check(other, w2, m2, offs2, ref2)
