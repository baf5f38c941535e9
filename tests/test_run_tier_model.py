"""CPU test of the clustering kernel's run tier (`run_clusters`), written as a
sequential model of its bitmap and its neighbour rule: rows of ceil(C / 32)
words, runs that end at word boundaries and are numbered in word order, each
run's contacts (a range of runs of the row above, with the runs beside it
across a word's edge, and the run that ends the word to its left).  The
labels must be the oracle's for module widths around the word size and any
density.  This checks the index arithmetic on CPU; the kernel itself is
compared with the oracle by the GPU tests."""
import numpy as np
import pytest

from oracle import oracle
from paper_2004_04334_gb300 import synth

FULL = 0xFFFFFFFF


def _clz(x):
    return 32 - int(x).bit_length()


def _popc(x):
    return bin(x).count("1")


def _model(rows, cols, R, C, rng):
    """Cluster id (smallest linear index) of every pixel."""
    W = (C + 31) // 32
    words = [0] * (R * W + 1)  # (one past the end is read and not used)
    for r, c in zip(rows, cols):
        words[r * W + (c >> 5)] |= 1 << (c & 31)
    heads = [x & ~(x << 1) & FULL for x in words]
    pre = np.concatenate([[0], np.cumsum([_popc(h) for h in heads])]).astype(int)
    nruns = pre[R * W]

    def run_of(r, c):
        b = 1 << (c & 31)
        return pre[r * W + (c >> 5)] + _popc(heads[r * W + (c >> 5)] & (b | (b - 1))) - 1

    pos = [None] * nruns
    for r, c in zip(rows, cols):
        if heads[r * W + (c >> 5)] >> (c & 31) & 1:
            pos[run_of(r, c)] = (r, c)
    parent = list(range(nruns))

    def find(x):
        while parent[x] != x:
            x = parent[x]
        return x

    for i in rng.permutation(nruns):
        r, c = pos[i]
        cw, b, wi = c >> 5, c & 31, r * W + (c >> 5)
        ln = _clz(int(f"{~(words[wi] >> b) & FULL:032b}"[::-1], 2))
        k = end = 0
        left_edge, right_edge = b == 0 and cw != 0, b + ln == 32 and cw + 1 < W
        if r > 0:
            wu = wi - W
            mask = (FULL >> (32 - ln)) << b
            t = words[wu] & (mask | mask << 1 | mask >> 1) & FULL
            if t:
                k = pre[wu] + _popc(heads[wu] & (t ^ (t - 1))) - 1
                end = pre[wu] + _popc(heads[wu] & (FULL >> _clz(t)))
            if left_edge and words[wu - 1] >> 31:
                end = end or pre[wu]
                k = pre[wu] - 1
            if right_edge and words[wu + 1] & 1:
                k = k if end else pre[wu + 1]
                end = pre[wu + 1] + 1
        touching = list(range(k, end))
        if left_edge and words[wi - 1] >> 31:
            touching.append(i - 1)
        for j in touching:
            a, x = find(i), find(j)
            parent[max(a, x)] = min(a, x)
    out = []
    for r, c in zip(rows, cols):
        rr, cc = pos[find(run_of(r, c))]
        out.append(rr * C + cc)
    return out


@pytest.mark.parametrize("C", [1, 2, 31, 32, 33, 63, 64, 65, 97, 416])
@pytest.mark.parametrize("density", [0.03, 0.3, 0.7, 1.0])
def test_run_model_matches_the_oracle(C, density):
    rng = np.random.default_rng(C * 100 + int(density * 10))
    R = 12
    lin = np.flatnonzero(rng.random(R * C) < density)
    rng.shuffle(lin)
    rows, cols = lin // C, lin % C
    gain, ped = np.array([70], np.int32), np.array([0], np.int32)
    ref = oracle.reconstruct_event(synth.pack(rows, cols, np.full(len(lin), 100)), np.zeros(len(lin), np.uint16), 1,
                                   gain, ped, rows=R, cols=C)
    assert np.array_equal(_model(rows.tolist(), cols.tolist(), R, C, rng), ref.label)
