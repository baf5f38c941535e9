"""GPU test: the stage timers name the kernels that ran, and no other."""
import numpy as np
import pytest

from paper_2004_04334_gb300 import hp, synth

pytestmark = pytest.mark.gpu

SMALL, MEDIUM = {"bucket", "cc", "finish"}, {"hist", "scan", "scatter", "cc", "finish"}
LARGE = {"hist", "scan", "scatter", "cc", "offsets", "copy"}
# modules, digis of each event, hash store, kernels
CASES = [(64, [1300], False, SMALL), (64, [0], False, {"scan", "cc", "finish"}), (64, [200000], False, MEDIUM),
         (64, [40] * 300, False, LARGE), (300, [2600000], False, LARGE - {"scatter"} | {"scatter_wide"}),
         (64, [64000], True, {"bucket", "cc_hash", "finish"}), (64, [3000000], True, LARGE - {"cc"} | {"cc_hash"})]


@pytest.mark.parametrize("M,sizes,hash_store,kernels", CASES)
def test_stage_timers_name_the_kernels_that_ran(M, sizes, hash_store, kernels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(len(sizes))
    E, N = len(sizes), sum(sizes)
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    key = np.concatenate([rng.choice(M * 66560, size=n, replace=False) for n in sizes])
    words = synth.pack(key % 66560 // 416, key % 416, rng.integers(1, 256, N)).astype(np.uint32)
    mods = (key // 66560).astype(np.uint16)
    with hp.Context(M, *synth.calibration(M, 5)) as ctx:
        if hash_store:
            ctx.set_tuning(E, N, next(t for t in ctx.tuning_candidates() if t["label_store"] == hp.HP_STORE_HASH))
        ctx.profile_enable(3)
        for _ in range(3):
            ev = ctx.enqueue_batch(words, mods, offs)
            assert ev.wait(60) == hp.HP_OK
            ev.release()
        got = ctx.profile_read()
        assert ctx.stats()["kernel_launches"] == 3 * len(kernels)
        ctx.profile_enable(0)
    assert list(got)[:6] == [f"{k}_kernel" for k in ("hist", "scan", "scatter", "cc", "offsets", "copy")]
    assert {k: n for k, (n, _) in got.items() if n} == {f"{k}_kernel": 3 for k in kernels}
    assert all((ms > 0) == (n > 0) for n, ms in got.values())
