"""Sizes of the clustering launches, worked out on the host (hp_internal.h):
the run tier's blocks fit wherever the hash store's do, so that every tile a
module size takes with one label store it takes with the other."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SM, OPT_IN, RESERVED = 228 * 1024, 227 * 1024, 1024  # shared memory of an SM, of a block at most, taken by each block
HASH_STATIC = 608                                    # static shared memory of the kernels
RUN_STATIC = {(1, 4): 6400, (2, 2): 3200, (2, 3): 3648, (3, 1): 1600}  # by blocks an SM and groups a block


def host_program(tmp_path, body):
    """The output of a host program of `body` with the kernels' header."""
    cxx = shutil.which("g++")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/x/x"))), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text('#include <cstdio>\n#include "hp_internal.h"\nint main() {\n' + body + "\nreturn 0; }\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2004_04334_gb300", "csrc"), "-I", inc,
                    str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def _hash_tile(rows, cols, blocks):
    """The largest tile with which `blocks` hash-store blocks stay on an SM."""
    most = min(OPT_IN - HASH_STATIC, SM // blocks - RESERVED - HASH_STATIC)
    return min(16384 if blocks == 1 else 4096, (most - (rows * cols + 31) // 32 * 12) // 20 // 256 * 256)


def test_the_run_tier_fits_every_tile_the_hash_store_fits(tmp_path):
    cases = []
    for rows in (1, 5, 9, 16, 31, 64, 80, 100, 128, 160, 173, 200, 255, 256):
        for cols in (1, 15, 31, 32, 33, 52, 64, 65, 97, 129, 200, 257, 320, 340, 345, 385, 416, 481, 512):
            if _hash_tile(rows, cols, 2) < 4096:
                continue  # refused by hp_create
            cases += [(rows, cols, _hash_tile(rows, cols, b), b, g) for b, g in RUN_STATIC]
    body = "\n".join(f'printf("%zu\\n", hp::run_smem_bytes({r}, {c}, {t}, {g}));' for r, c, t, b, g in cases)
    for (r, c, t, b, g), got in zip(cases, map(int, host_program(tmp_path, body).split())):
        need = got + RUN_STATIC[b, g]
        assert need <= OPT_IN and b * (need + RESERVED) <= SM, (r, c, t, b, g)


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols", [(16, 32), (80, 52), (160, 100), (160, 416)])
def test_the_largest_tiles_are_accepted_and_exact(rows, cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle
    from paper_2004_04334_gb300 import hp, synth
    from tests.gpu_util import assert_batch_matches

    rng = np.random.default_rng(rows)
    M, px = 6, rows * cols
    lin = [rng.choice(px, size=max(1, int(f * px)), replace=False) for f in (0.01, 0.1, 0.25, 0.5, 0.8, 1.0)]
    words = np.concatenate([synth.pack(x // cols, x % cols, rng.integers(20, 256, len(x))) for x in lin]).astype(np.uint32)
    mods = np.concatenate([np.full(len(x), i, np.uint16) for i, x in enumerate(lin)])
    offs = np.array([0, len(words)], np.uint64)
    gain, ped = np.full(M, 70, np.int32), np.full(M, 50, np.int32)
    ref = oracle.reconstruct_batch(words, mods, offs, M, gain, ped, rows=rows, cols=cols)
    with hp.Context(M, gain, ped, rows=rows, cols=cols) as ctx:
        for blocks in (1, 2, 3):
            for store, threads in ((hp.HP_STORE_BITMAP, 512), (hp.HP_STORE_HASH, 256)):
                t = {"tile_slots": _hash_tile(rows, cols, blocks), "blocks_per_sm": blocks, "ticket_items": 4,
                     "warp_max": 64, "label_store": store, "item_threads": threads}
                assert ctx.try_set_tuning(1, len(words), t) == hp.HP_OK, t
                ev = ctx.enqueue_batch(words, mods, offs, flags=hp.HP_WANT_LABELS)
                ev.wait(60)
                assert_batch_matches(ev.fetch(), ref, offs)
                ev.release()
