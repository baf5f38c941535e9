"""Performance cases of libhp: what a reconstruction program has it do, through its public entry points.

A case names a synthetic recipe (the detector's size, the events and their mean digis) and the entry point its events go
through:

``device``      Context.reconstruct_device on the current stream: inputs and outputs stay in device memory (with ``hits``
                followed by Context.hits_device, the next module of a GPU chain)
``graph``       the same pass captured once and replayed (Context.graph_capture, Graph.launch)
``host_event``  Context.enqueue_event, wait, fetch: one event from pageable host memory to the program's own arrays
``host_batch``  Context.enqueue_batch from pinned memory, wait, fetch: the clusters into the program's arrays, the compact
                labels where the library put them
``serve``       Context.submit of a burst of events (read in place from pinned memory) to the serving loop, then each one's
                clusters into the program's arrays

Recipes (paper_2004_04334_gb300.synth): ``blobs`` is the 64-module recipe of the batched and serving workloads, ``sparse``
the full-detector recipe, ``noisy`` the same with 1% noise occupancy, ``dense`` the high-occupancy one with streaks and hot
modules.  Events of a batch have equal expected sizes (``spread`` "even"), sizes uniform within a factor of 20 ("uniform")
or lognormal ones as a trigger farm sees them ("lognormal").  The sizes follow from the case, the digis from the seed.
"""
import atexit
import math
import os
from concurrent.futures import ThreadPoolExecutor
from dataclasses import replace

import numpy as np
import torch

from paper_2004_04334_gb300 import hp, synth

ROWS, COLS = synth.ROWS, synth.COLS
PIXEL_THR, CLUSTER_THR = 1000, 4000
DENSE_DIGIS = synth.OCCUPANCY.expected_digis() / synth.OCCUPANCY.n_modules  # of a module of the dense recipe
NOISY_DIGIS = synth.FULL_LITERAL.expected_digis() / synth.FULL_LITERAL.n_modules


def _case(name, entry, recipe, modules, events, digis, spread="even", hits=False, tuned=False):
    c = {"entry": entry, "recipe": recipe, "modules": modules, "events": events, "digis": digis, "spread": spread,
         "hits": hits, "tuned": tuned}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one event of the 64-module set-up, kept on the device; launch latency
        _case("event_small", "device", "blobs", 64, 1, 1300),
        # one event of the whole detector (1856 modules, ~60k digis), kept on the device for the next module
        _case("event_full", "device", "sparse", 1856, 1, 60000),
        # the same event as a host program sees it: copied in, reconstructed with labels, copied out
        _case("event_full_host", "host_event", "sparse", 1856, 1, 60000),
        # one event with 1% noise in every module (1.5M digis): the largest single event
        _case("event_noisy", "device", "noisy", 1856, 1, int(1856 * NOISY_DIGIS)),
        # full-detector events in a fixed-shape batch, replayed as a graph: many small items
        _case("batch_full_graph", "graph", "sparse", 1856, 16, 60000),
        # a serving-size batch (lognormal event sizes) and its hits: the raw -> clusters -> hits chain
        _case("chain_lognormal", "device", "blobs", 64, 48, 100000, spread="lognormal", hits=True),
        # the benchmark's batch: 256 uneven events, on the device, with the launch settings autotuned
        _case("batch_mixed", "device", "blobs", 64, 256, 105000, spread="uniform", tuned=True),
        # a batch from pinned host memory and back, compact labels: the host link and the kernels behind it
        _case("batch_mixed_host", "host_batch", "blobs", 64, 64, 105000, spread="uniform"),
        # high-occupancy events (streaks, hot modules at 20%): large items, autotuned
        _case("batch_dense", "device", "dense", 1856, 8, int(1856 * DENSE_DIGIS), tuned=True),
        # a burst of requests to the serving loop
        _case("serve_burst", "serve", "blobs", 64, 16, 100000, spread="lognormal"),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: an entry, a recipe and sizes spread over what the listed cases span."""
    entry = rng.choice(["device", "device", "device", "graph", "host_event", "host_batch", "serve"])
    recipe = rng.choice(["blobs", "blobs", "sparse", "noisy", "dense"]) if entry != "serve" else "blobs"
    tuned = entry == "device" and rng.random() < 0.3
    if recipe == "blobs":  # 20 to 8,000 digis a module
        modules = rng.choice([64, _between(rng, 16, 256)])
        digis = _between(rng, 20 * modules, min(500000, 8000 * modules))
    elif recipe == "sparse":  # a few to a hundred digis a module
        modules = rng.choice([1856, _between(rng, 100, 1856)])
        digis = _between(rng, 8 * modules, 100 * modules)
    else:
        modules = _between(rng, 16, 1856)
        digis = int(modules * (NOISY_DIGIS if recipe == "noisy" else DENSE_DIGIS) * rng.uniform(0.3, 1.0))
    most = {"device": 20e6, "graph": 20e6, "host_event": 2e6, "host_batch": 6e6, "serve": 1.5e6}[entry]
    limit = max(1, min(256 if entry != "serve" else 16, int(most / digis)))
    events = 1 if entry == "host_event" or rng.random() < 0.25 else _between(rng, 1, limit)
    if digis > most:  # one event past the entry's range: fewer digis a module
        digis = int(most)
    spread = rng.choice(["even", "uniform", "lognormal"]) if events > 1 and recipe == "blobs" else "even"
    return _case(None, entry, recipe, modules, events, digis, spread, entry == "device" and rng.random() < 0.3, tuned)


# ------------------------------------------------------------------ inputs

def _recipe(case, digis):
    M = case["modules"]
    if case["recipe"] == "blobs":
        noise = min(synth.TINY.lambda_noise, 0.1 * digis / M)
        return replace(synth.TINY, n_modules=M, lambda_noise=noise, lambda_clusters=(digis / M - noise) / 6.5)
    if case["recipe"] == "sparse":
        inner = min(synth.FULL.n_inner, M // 8)
        return replace(synth.FULL, n_modules=M, n_inner=inner, lambda_noise=0.01 * digis / M,
                       lambda_clusters=0.99 * digis / ((M + 3 * inner) * 10.5))
    if case["recipe"] == "noisy":
        f = digis / (M * NOISY_DIGIS)
        base = synth.FULL_LITERAL
        return replace(base, n_modules=M, n_inner=min(base.n_inner, M // 8),
                       lambda_noise=f * base.lambda_noise, lambda_clusters=f * base.lambda_clusters)
    f = digis / (M * DENSE_DIGIS)
    base = synth.OCCUPANCY
    return replace(base, n_modules=M, lambda_clusters=f * base.lambda_clusters, hot_frac=f * base.hot_frac)


def _sizes(case):
    """Digis of each event."""
    rng = np.random.default_rng(case["events"])
    E, mean = case["events"], float(case["digis"])
    if case["spread"] == "uniform":
        sizes = rng.uniform(2 * mean / 21, 40 * mean / 21, E)
    elif case["spread"] == "lognormal":
        sizes = np.minimum(rng.lognormal(math.log(mean) - 0.32, 0.8, E), 5 * mean)
    else:
        sizes = np.full(E, mean)
    return np.maximum(1, sizes.astype(np.int64))


def _event(case, size, seed):
    """`size` digis: an event of a little more, cut (its digis are in random order)."""
    more = size + 4 * math.sqrt(30 * size)
    while True:
        words, mods = synth.make_event(_recipe(case, more), seed)
        if len(words) >= size:
            return words[:size], mods[:size]
        more *= 1.1
        seed += 1


def _events(case, seed):
    """Words uint32[N], module ids uint16[N] and offsets uint64[E + 1] of the case's events."""
    sizes = _sizes(case)
    seeds = np.random.default_rng(seed).integers(0, 2**62, len(sizes))
    with ThreadPoolExecutor(min(len(sizes), os.cpu_count() or 1)) as pool:
        made = list(pool.map(lambda a: _event(case, int(a[0]), int(a[1])), zip(sizes, seeds)))
    offsets = np.zeros(len(sizes) + 1, np.uint64)
    offsets[1:] = np.cumsum(sizes)
    return np.concatenate([w for w, _ in made]), np.concatenate([m for _, m in made]), offsets


_contexts = {}


def _calibration(M):
    return synth.calibration(M, 2004)


def _context(M, use):
    """The program's context for a detector of M modules (made once, as such a program does)."""
    if (M, use) not in _contexts:
        gain, ped = _calibration(M)
        ctx = hp.Context(M, gain, ped, pixel_thr=PIXEL_THR, cluster_thr=CLUSTER_THR)
        ctx.set_geometry(*synth.barrel_geometry(M), synth.PITCH_ROW, synth.PITCH_COL)
        if use == "serve":
            ctx.serve_start(max_batch_events=16, max_batch_digis=1 << 22, nocopy=True)
        _contexts[M, use] = ctx
    return _contexts[M, use]


@atexit.register
def _close():
    for ctx in _contexts.values():
        ctx.close()
    _contexts.clear()


def _dev(a):
    t = {np.dtype(np.uint64): np.int64, np.dtype(np.uint32): np.int32, np.dtype(np.uint16): np.int16}[a.dtype]
    return torch.from_numpy(a.view(t)).cuda()


class _State:
    """What the program holds: its inputs, output arrays, and a product or a graph to give back."""

    def __init__(self, case):
        self.entry, self.hits = case["entry"], case["hits"]
        self.product = self.graph = None

    def __del__(self):
        if _contexts and self.product is not None:
            self.product.release()
        if _contexts and self.graph is not None:
            self.graph.destroy()


def prepare(case, seed):
    s = _State(case)
    words, mods, offsets = _events(case, seed)
    use = s.entry if s.entry == "serve" else "tuned" if case["tuned"] else "plain"
    s.ctx = _context(case["modules"], use)
    s.E, s.N = case["events"], int(offsets[-1])
    if s.entry in ("device", "graph"):
        s.inputs = [_dev(offsets), _dev(words), _dev(mods)]
        s.out = hp.DeviceOutputs(s.E, s.N, "cuda")
        s.cols = {k: getattr(s.out, k) for k in ("module", "id", "charge", "npix", "x", "y")}
        if s.hits:
            s.cols.update({k: torch.empty_like(s.out.x) for k in ("hx", "hy", "hz")})
        for t in s.cols.values():  # what no cluster reaches stays zero
            t.zero_()
        s.result = dict(s.cols, cluster_offsets=s.out.cluster_offsets, event_status=s.out.event_status,
                        label=s.out.label)
        s.args = (s.E, s.N, *[t.data_ptr() for t in s.inputs], s.out)
        if case["tuned"]:
            s.ctx.autotune(*s.args)
        if s.entry == "graph":
            s.graph = s.ctx.graph_capture(*s.args)
    else:
        # pinned inputs, where the library reads them in place; the program's own arrays take the results
        words, mods = (torch.from_numpy(a.view(t)) for a, t in ((words, np.int32), (mods, np.int16)))
        s.offsets = offsets
        s.inputs = [words, mods] if s.entry == "host_event" else [words.pin_memory(), mods.pin_memory()]
        w, m = (t.numpy().view(v) for t, v in zip(s.inputs, (np.uint32, np.uint16)))
        s.ranges = [(int(a), int(b)) for a, b in zip(offsets[:-1], offsets[1:])]
        s.events = [(w[a:b], m[a:b]) for a, b in s.ranges]
        s.cols = {k: torch.zeros(s.N, dtype=torch.float32 if k in "xy" else torch.int32)
                  for k in ("module", "id", "charge", "npix", "x", "y")}
        s.result = dict(s.cols, cluster_offsets=np.zeros(s.E + 1, np.int64), event_status=np.zeros(s.E, np.int32))
        if s.entry == "host_event":
            s.result["label"] = torch.zeros(s.N, dtype=torch.int32)
    return s


def _take(s, res, at=0):
    """Copy a product's clusters into the program's arrays, from position `at` on."""
    n = len(res.id)
    for k, t in s.cols.items():
        v = getattr(res, k)
        t[at:at + n].copy_(torch.from_numpy(v.view(np.int32) if v.dtype == np.uint32 else v))


def run(s):
    if s.entry == "graph":
        s.graph.launch(torch.cuda.current_stream().cuda_stream)
        return s.result
    if s.entry == "device":
        stream = torch.cuda.current_stream().cuda_stream
        s.ctx.reconstruct_device(*s.args, stream)
        if s.hits:
            c = s.cols
            s.ctx.hits_device(s.E, s.N, s.out.cluster_offsets.data_ptr(), *[c[k].data_ptr() for k in
                              ("module", "x", "y", "hx", "hy", "hz")], stream)
        return s.result
    if s.entry == "serve":
        for e, ev in enumerate([s.ctx.submit(*ev) for ev in s.events]):
            ev.wait()
            res = ev.fetch(copy=False)
            _take(s, res, s.ranges[e][0])
            s.result["cluster_offsets"][e + 1] = len(res.id)
            s.result["event_status"][e] = res.status
            ev.release()
        return s.result
    if s.entry == "host_event":
        ev = s.ctx.enqueue_event(*s.events[0], flags=hp.HP_WANT_LABELS)
    else:
        if s.product is not None:  # done with the last batch's labels
            s.product.release()
        ev = s.product = s.ctx.enqueue_batch(*s.inputs, s.offsets, flags=hp.HP_INPUT_NOCOPY | hp.HP_LABELS_U16)
    ev.wait()
    res = ev.fetch(copy=False)
    _take(s, res)
    s.result["cluster_offsets"][:] = res.cluster_offsets
    s.result["event_status"][:] = res.event_status
    if s.entry == "host_event":
        s.result["label"].copy_(torch.from_numpy(res.label))
        ev.release()
        return s.result
    return dict(s.result, label16=res.label16.view(np.int16), item_first=res.item_first.view(np.int32))


def work(case):
    """Words, module ids, offsets and calibration in; a label a digi (not from the serving loop) and 24 bytes a cluster (one per 7.5 digis) out.
    Operations: calibration, threshold and four sums a digi."""
    E, N, M = case["events"], int(_sizes(case).sum()), case["modules"]
    clusters = N / 7.5
    label = {"host_batch": 2 * N + 4 * E * M, "serve": 0}.get(case["entry"], 4 * N)
    hits = 24 * clusters if case["hits"] else 0
    return {"bytes": 6 * N + 16 * (E + 1) + 8 * M + label + 24 * clusters + hits, "flops": 9 * N}


# ------------------------------------------------------------------ results in 64 bits

def _centroids(words, mods, offsets, M):
    """Module, event, x and y of the kept clusters, in (event, module, id) order: plain torch, 64 bits."""
    gain, ped = (torch.from_numpy(a.astype(np.int64)).cuda() for a in _calibration(M))
    w = torch.from_numpy(words.astype(np.int64)).cuda()
    m = torch.from_numpy(mods.astype(np.int64)).cuda()
    ev = torch.repeat_interleave(torch.arange(len(offsets) - 1), torch.from_numpy(np.diff(offsets.astype(np.int64)))).cuda()
    row, col, adc = w & 255, (w >> 8) & 511, (w >> 17) & 255
    q = adc * gain[m] - ped[m]
    keep = q >= PIXEL_THR
    width = COLS + 1  # a free column between rows
    key = (((ev * M + m) * (ROWS + 1) + row) * width + col)[keep]
    key, order = torch.sort(key)
    q, row, col, item = q[keep][order], row[keep][order], col[keep][order], (ev * M + m)[keep][order]
    n = len(key)
    label = torch.arange(n, device=key.device)
    edges = []
    for d in (1, width - 1, width, width + 1):  # left, upper right, upper, upper left
        at = torch.searchsorted(key, key - d).clamp(max=max(n - 1, 0))
        hit = (key[at] == key - d) if n else at.bool()
        if d != 1:
            hit &= row > 0
        edges.append((torch.nonzero(hit).squeeze(1), at[hit]))
    a, b = (torch.cat([e[i] for e in edges]) for i in range(2))
    while n:
        low = torch.minimum(label[a], label[b])
        new = label.clone()
        new.scatter_reduce_(0, a, low, "amin")
        new.scatter_reduce_(0, b, low, "amin")
        new.scatter_reduce_(0, label[a], low, "amin")
        new.scatter_reduce_(0, label[b], low, "amin")
        new = new[new]
        if torch.equal(new, label):
            break
        label = new
    roots, inverse = torch.unique(label, return_inverse=True)
    total, mr, mc = (torch.zeros(len(roots), dtype=torch.int64, device=key.device).index_add_(0, inverse, v)
                     for v in (q, q * row, q * col))
    good = total >= CLUSTER_THR
    x, y = mr[good].double() / total[good].double(), mc[good].double() / total[good].double()
    return (item[roots][good] % M).cpu().numpy(), (item[roots][good] // M).cpu().numpy(), x.cpu().numpy(), y.cpu().numpy()


def exact(case, seed):
    words, mods, offsets = _events(case, seed)
    M, N = case["modules"], len(words)
    module, event, x, y = _centroids(words, mods, offsets, M)
    at = np.arange(len(x))  # positions in the output arrays, which are as long as the input
    if case["entry"] == "serve":
        at += (offsets[event].astype(np.int64) - np.searchsorted(event, event))
    cols = {"x": x, "y": y}
    if case["hits"]:
        origin, rot = (a.astype(np.float64) for a in synth.barrel_geometry(M))
        u, v = (x - (ROWS - 1) / 2) * synth.PITCH_ROW, (y - (COLS - 1) / 2) * synth.PITCH_COL
        for i, k in enumerate(("hx", "hy", "hz")):
            cols[k] = origin[module, i] + rot[module, i, 0] * u + rot[module, i, 1] * v
    out = dict.fromkeys(("cluster_offsets", "event_status", "module", "id", "charge", "npix"))
    for k, a in cols.items():
        out[k] = np.zeros(N)
        out[k][at] = a
    if case["entry"] != "serve":
        out.update(dict.fromkeys(("label16", "item_first") if case["entry"] == "host_batch" else ("label",)))
    return out
