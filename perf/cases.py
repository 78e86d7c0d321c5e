"""The calls this GGArray is used for, as cases that can be timed and compared.

A case is a dict of plain values: the kind of work, the array's shape (L
LFVectors of T-thread blocks, first bucket B elements, E-byte elements) and
the sizes of the call.  `prepare` makes what a program holds before the
call, `run` makes one pass through the public entry points and returns
everything the pass computes.  All results are whole numbers (elements,
offsets) or records copied bit for bit, so `exact` has nothing to add.

The kinds:

step       every operation once, in the order of the paper's experiments:
           clear, insert, random reads, random writes, the two +1 sweeps
           (rw_b, rw_g), flatten.
grow       counts and values from device memory: clear, insert R rounds,
           flatten, prefix sum of the LFVector sizes.
read       random (or ascending) global indices read from a grown array.
write      the same, written, then the flattened result.
sweep      the r/w operation by block structure and by global index, then
           the flattened result.
generated  insertion whose counts and values the inserting threads draw,
           by the batched-rounds kernel or (push) by one push per round
           through the device API; then flatten.
expand     pushes of values read from device memory through the device API,
           then flatten.
batch      many arrays of uneven size grown by one graph replay, 4096 reads
           from each, 16 of them flattened.
serve      one step of a request server: appends to many arrays of one pool,
           4096 reads from each, the retired ones flattened.
two_phase  records spawn children generation by generation, are flattened,
           and updated by streaming passes over the contiguous copy.
"""

import ctypes
import math

import torch

from paper_2209_00103_gb300 import batching, gga
from paper_2209_00103_gb300 import workloads as wl

MEAN = {"bernoulli": 0.5, "uniform3": 1.0, "geometric": 1.0, "poisson": 1.0}   # elements per thread and round
COEFFS = (1, 1 << 20, 1 << 19)   # value = gtid + round * 2^20 + k * 2^19: tells where it was inserted


def listed():
    return [
        # The smallest program: the paper's tiny array, every operation once.
        # Launches and host calls are all there is.
        dict(name="step_tiny", kind="step", L=32, T=256, B=1024, E=4, R=10, dist="bernoulli", n=4096),
        # The headline insertion: 2^28 int32 elements in 512 rounds into 1024
        # LFVectors, and the flatten that ends the insertion phase.
        dict(name="grow_paper", kind="grow", L=1024, T=512, B=4096, E=4, R=512, dist="uniform3"),
        # 16-byte records (particles, key-value pairs) with shapes that are
        # not powers of two: ragged tiles everywhere.
        dict(name="grow_records_ragged", kind="grow", L=301, T=200, B=256, E=16, R=61, dist="poisson"),
        # Random access to the paper-sized array, as between its insertions.
        dict(name="read_paper", kind="read", L=1024, T=512, B=4096, E=4, R=512, n=1 << 26, order="uniform"),
        dict(name="write_paper", kind="write", L=1024, T=512, B=4096, E=4, R=512, n=1 << 26, order="uniform"),
        # The r/w operation over the paper-sized array, both ways.
        dict(name="sweep_paper", kind="sweep", L=1024, T=512, B=4096, E=4, R=512, repeats=1),
        # Insertion from inside an application kernel, by batched rounds.
        dict(name="generated_paper", kind="generated", L=1024, T=512, B=4096, E=4, R=512, dist="uniform3", push=False),
        # The same as Algorithm 1 states it: one push per round (device API).
        dict(name="push_paper", kind="generated", L=1024, T=512, B=4096, E=4, R=512, dist="uniform3", push=True),
        # A user kernel that reads its elements from memory and pushes them.
        dict(name="expand_paper", kind="expand", L=1024, T=512, B=4096, E=4, R=512, dist="uniform3"),
        # Many arrays of uneven size (lognormal, median 64K elements) and mixed
        # payloads grown together.
        dict(name="batch_lognormal", kind="batch", arrays=1024),
        # One step of the request server at a high load.
        dict(name="serve_step", kind="serve", arrays=256, L=4, B=1024, E=8, most=1_000_000, retire=16),
        # The two-phase case study: 2^20 records, 8 generations (2^28 records).
        dict(name="two_phase_8", kind="two_phase", L=1024, T=512, B=4096, n0=1 << 20, generations=8, passes=2),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _shape(rng, most_elems, E=None, max_t=1024):
    """L, T, B, E, R with up to most_elems elements (and bytes as int32 ones)."""
    E = E or rng.choice((4, 4, 8, 16))
    total = _log(rng, 20_000, most_elems * 4 // E)
    T = rng.choice((32, 128, 256, 512, max_t, _log(rng, 17, max_t)))
    L = _log(rng, 16, max(16, min(2048, total // (2 * T))))
    R = max(1, min(2048, total // (L * T)))
    per = max(16, T * R)
    B = 1 << int(round(math.log2(max(16, min(65536, per / rng.choice((1, 4, 16, 64)))))))
    return dict(L=L, T=T, B=B, E=E, R=R)


def draw(rng):
    kind = rng.choice(("step", "grow", "read", "write", "sweep", "generated", "expand", "batch", "serve", "two_phase"))
    most = 1 << 27
    if kind == "step":
        c = _shape(rng, 1 << 26, E=rng.choice((4, 8)))
        return dict(kind=kind, **c, dist=rng.choice(("bernoulli", "uniform3", "poisson")),
                    n=_log(rng, 1000, max(1000, c["L"] * c["T"] * c["R"] // 4)))
    if kind == "grow":
        return dict(kind=kind, **_shape(rng, most), dist=rng.choice(("bernoulli", "uniform3", "geometric", "poisson")))
    if kind in ("read", "write"):
        return dict(kind=kind, **_shape(rng, 1 << 28), n=_log(rng, 4096, 1 << 25),
                    order=rng.choice(("uniform", "uniform", "ascending")))
    if kind == "sweep":
        return dict(kind=kind, **_shape(rng, 1 << 28, E=rng.choice((4, 4, 8))), repeats=rng.choice((1, 1, 30)))
    if kind == "generated":
        return dict(kind=kind, **_shape(rng, most), dist=rng.choice(("bernoulli", "uniform3", "geometric", "poisson")),
                    push=rng.random() < 0.4)
    if kind == "expand":
        return dict(kind=kind, **_shape(rng, most, max_t=512), dist=rng.choice(("bernoulli", "uniform3", "poisson")))
    if kind == "batch":
        return dict(kind=kind, arrays=_log(rng, 16, 1000))
    if kind == "serve":
        return dict(kind=kind, arrays=_log(rng, 16, 480), L=rng.choice((1, 3, 4, 8)), B=rng.choice((256, 1024, 4096)),
                    E=rng.choice((4, 8, 8, 16)), most=_log(rng, 1000, 1_000_000), retire=rng.choice((1, 4, 16)))
    n0 = _log(rng, 1 << 14, 1 << 19)
    return dict(kind=kind, L=_log(rng, 16, n0 // 256), T=rng.choice((128, 256, 512)), B=rng.choice((256, 1024, 4096)),
                n0=n0, generations=rng.randrange(1, 9), passes=rng.choice((1, 2, 4)))


# ---------------------------------------------------------------------------


def _need(L, B, E, size):
    """Bytes of the buckets that L LFVectors of up to `size` elements reach."""
    cap = total = 0
    while cap < size:
        total += max(256, (cap + B) * E)
        cap = 2 * cap + B
    return L * total + (1 << 20)


def _largest(c, dist):
    """A size no LFVector of T * R draws exceeds (eight standard deviations)."""
    n = c["T"] * c["R"]
    return int(n * MEAN[dist] + 8 * math.sqrt(2 * n)) + 64


def _array(c, dist="uniform3"):
    return gga.GGArray(c["L"], c["T"], c["B"], c["E"], _need(c["L"], c["B"], c["E"], _largest(c, dist)))


def _flat(c, dist="uniform3"):
    """A destination for the flattened array, whatever its size turns out to be."""
    return gga.elem_tensor(c["L"] * _largest(c, dist), c["E"]).zero_()


def _insert_spec(c, seed):
    return wl.InsertSpec(L=c["L"], T=c["T"], E=c["E"], seed=seed + 1, dist=c["dist"], rounds=c["R"], coeffs=COEFFS)


def _gen_spec(c, seed, dist):
    thr = wl.poisson1_thresholds() if dist == "poisson" else None
    return gga.make_gen_spec(seed + 1, dist, COEFFS, thresholds=thr)


def _size(g):
    n, rc = g.size()
    assert rc == gga.GGA_OK, rc
    return n


def _grown(c, seed):
    g = _array(c)
    g.insert_generated(_gen_spec(c, seed, "uniform3"), c["R"])
    return g, _size(g)


def _indices(c, seed, N):
    idx = wl.uniform_indices_t(seed + 2, c["n"], N, "cuda")
    return idx.sort().values if c.get("order") == "ascending" else idx


class _State:
    pass


def prepare(case, seed):
    s, c, kind = _State(), case, case["kind"]
    s.case, s.kind = c, kind
    if kind in ("step", "grow"):
        s.counts, s.values = wl.make_insert_inputs_t(_insert_spec(c, seed), "cuda")
        N = s.values.shape[0]
        s.g = _array(c, c["dist"])
        s.flat = _flat(c, c["dist"])
        s.offsets = torch.empty(c["L"] + 1, dtype=torch.int64, device="cuda")
        if kind == "step":
            s.idx, s.at = _indices(c, seed, N), _indices(c, seed + 7, N)
            s.vals = wl.index_keyed_values_t(seed + 3, s.at, c["E"])
            s.out = gga.elem_tensor(c["n"], c["E"])
    elif kind in ("read", "write"):
        s.g, N = _grown(c, seed)
        s.idx = _indices(c, seed, N)
        if kind == "read":
            s.out = gga.elem_tensor(c["n"], c["E"])
        else:
            s.vals = wl.index_keyed_values_t(seed + 3, s.idx, c["E"])
            s.flat = _flat(c)
    elif kind == "sweep":
        s.g, _ = _grown(c, seed)
        s.flat = _flat(c)
    elif kind == "generated":
        s.g, s.spec, s.flat = _array(c, c["dist"]), _gen_spec(c, seed, c["dist"]), _flat(c, c["dist"])
    elif kind == "expand":
        spec = _insert_spec(c, seed)
        r = torch.arange(c["R"], dtype=torch.int64, device="cuda")
        t = torch.arange(c["L"] * c["T"], dtype=torch.int64, device="cuda")
        h = wl.splitmix_at_t(spec.seed, (r[:, None] << 32) | t[None, :])
        s.counts = wl.draw_counts_t(c["dist"], h).reshape(c["R"], c["L"], c["T"])
        s.inputs = wl.expand_inputs_t(spec, "cuda")
        s.g, s.flat = _array(c, c["dist"]), _flat(c, c["dist"])
    elif kind == "batch":
        _prepare_batch(s, c, seed)
    elif kind == "serve":
        _prepare_serve(s, c, seed)
    else:
        _prepare_two_phase(s, c, seed)
    return s


def _prepare_batch(s, c, seed):
    sizes, rule = batching.batched_sizes(c["arrays"]), batching.tuned_rule()
    params = [batching.params_for(rule, a, int(n)) for a, n in enumerate(sizes)]
    E = [batching.payload_bytes(a) for a in range(len(sizes))]
    need = sum(_need(L, B, e, int(n) // L + 1) for n, (_, L, B), e in zip(sizes, params, E))
    s.pool = gga.GGAPool(need, 256 * 4)
    s.arrays = [gga.GGArray(L, T, B, e, shared_pool=s.pool) for (T, L, B), e in zip(params, E)]
    thr = wl.poisson1_thresholds()
    s.batch = gga.GGABatch([(g, gga.make_gen_spec(((seed + 3) << 32) | a, "poisson", (0x10001, 0x9E3779B9, 7),
                                                  thresholds=thr), int(n))
                            for a, (g, n) in enumerate(zip(s.arrays, sizes))])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    s.batch.capture(side)
    torch.cuda.current_stream().wait_stream(side)
    s.reads = torch.empty(sum(4096 * e for e in E) // 8, dtype=torch.int64, device="cuda")
    at = 0
    s.lookups = (gga.gga_read_req * len(E))()   # the request table, as include/gga.h declares it
    for a, g in enumerate(s.arrays):
        s.lookups[a].array, s.lookups[a].n, s.lookups[a].seed = g.h, 4096, seed + a
        s.lookups[a].out = s.reads.data_ptr() + at
        at += 4096 * E[a]
    s.lib = gga.load_library()
    step = max(1, len(sizes) // 16)
    s.flats = [(s.arrays[a], gga.elem_tensor(int(sizes[a]), E[a])) for a in range(0, len(sizes), step)][:16]


def _prepare_serve(s, c, seed):
    A, E = c["arrays"], c["E"]
    h = wl.splitmix_at(4, torch.arange(A).numpy())
    n = [int(math.exp((int(x) >> 11) / 2.0 ** 53 * math.log(c["most"]))) for x in h]
    s.pool = gga.GGAPool(sum(_need(c["L"], c["B"], E, m // c["L"] + 1) for m in n), 256)
    s.arrays = [gga.GGArray(c["L"], 256, c["B"], E, shared_pool=s.pool) for _ in range(A)]
    # The batch that empties the arrays at the start of a step.
    s.batch = gga.GGABatch([(g, gga.make_gen_spec(1, "bernoulli", (1, 0, 0)), m) for g, m in zip(s.arrays, n)])
    s.reads = gga.elem_tensor(A * 4096, E)
    # The server's request tables, as include/gga.h declares them.
    s.appends = (gga.gga_append_req * A)()
    s.lookups = (gga.gga_read_req * A)()
    for i, g in enumerate(s.arrays):
        s.appends[i].array, s.appends[i].n, s.appends[i].tag = g.h, n[i], (seed + i) & 0xFFFFFFFF
        s.lookups[i].array, s.lookups[i].n, s.lookups[i].seed = g.h, 4096, seed + i
        s.lookups[i].out = s.reads.data_ptr() + i * 4096 * E
    s.flats = [(s.arrays[a], gga.elem_tensor(n[a], E)) for a in range(0, A, max(1, A // c["retire"]))][:16]
    s.lib = gga.load_library()


def _prepare_two_phase(s, c, seed):
    L, n0 = c["L"], c["n0"]
    per = n0 / L * 2.0 ** c["generations"]
    most = int(per * (1 + 8 / math.sqrt(n0 / L))) + 64   # a size no LFVector reaches (eight standard deviations)
    s.g = gga.GGArray(L, c["T"], c["B"], 16, _need(L, c["B"], 16, most))
    s.counts = torch.from_numpy(wl.split_counts(L, c["T"], n0).view("int32")).cuda()
    s.records = wl.initial_records_t(n0, "cuda")
    s.seed = seed + 5
    _grow_two_phase(s)                     # how large the population gets: the work passes take it
    s.n = _size(s.g)
    s.flat = gga.elem_tensor(L * most, 16).zero_()
    s.offsets = torch.empty(L + 1, dtype=torch.int64, device="cuda")


def _grow_two_phase(s):
    s.g.clear()
    s.g.insert(s.counts, s.records)
    for gen in range(s.case["generations"]):
        gga.gga_twophase_spawn(s.g.h, gen, s.seed)


def run(s):
    g, kind = getattr(s, "g", None), s.kind
    if kind == "step":
        g.clear()
        g.insert(s.counts, s.values)
        g.read(s.idx, s.out)
        g.write(s.at, s.vals)
        g.sweep(gga.GGA_RW_B)
        g.sweep(gga.GGA_RW_G)
        g.flatten(s.flat)
        gga.gga_offsets(g.h, s.offsets)
        return s.out, s.flat, s.offsets
    if kind == "grow":
        g.clear()
        g.insert(s.counts, s.values)
        g.flatten(s.flat)
        gga.gga_offsets(g.h, s.offsets)
        return s.flat, s.offsets
    if kind == "read":
        return g.read(s.idx, s.out)
    if kind == "write":
        g.write(s.idx, s.vals)
        return g.flatten(s.flat)
    if kind == "sweep":
        g.sweep(gga.GGA_RW_B, 1, s.case["repeats"])
        g.sweep(gga.GGA_RW_G, 1, s.case["repeats"])
        return g.flatten(s.flat)
    if kind == "generated":
        g.clear()
        (g.push_generated if s.case["push"] else g.insert_generated)(s.spec, s.case["R"])
        return g.flatten(s.flat)
    if kind == "expand":
        g.clear()
        g.push_expand(s.counts, s.inputs)
        return g.flatten(s.flat)
    if kind in ("batch", "serve"):
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        if kind == "batch":
            s.batch.replay()
        else:
            s.batch.clear()
            assert s.lib.gga_append_batch(s.appends, len(s.appends), stream) == gga.GGA_OK
        assert s.lib.gga_read_batch(s.lookups, len(s.lookups), stream) == gga.GGA_OK
        return [s.reads] + [a.flatten(f) for a, f in s.flats]
    _grow_two_phase(s)
    g.flatten(s.flat)
    gga.gga_twophase_work(s.flat[:s.n], s.case["passes"])
    gga.gga_offsets(g.h, s.offsets)
    return s.flat, s.offsets


def work(case):
    c, kind = case, case["kind"]
    E = c.get("E", 16)
    slots = c["L"] * c["T"] * c.get("R", 1) if "T" in c else 0
    N = slots * MEAN[c.get("dist", "uniform3")]
    flatten = 2 * E * N
    if kind == "step":     # counts and values in, elements out; per access index, element, value; two sweeps
        b = 4 * slots + 2 * E * N + 2 * c["n"] * (8 + 2 * E) + 2 * 2 * E * N + flatten
    elif kind == "grow":
        b = 4 * slots + 2 * E * N + flatten
    elif kind == "read":
        b = c["n"] * (8 + 2 * E)
    elif kind == "write":
        b = c["n"] * (8 + 2 * E) + flatten
    elif kind == "sweep":
        b = 2 * 2 * E * N + flatten
    elif kind == "generated":
        b = E * N + flatten
    elif kind == "expand":
        b = (4 + E) * slots + E * N + flatten
    elif kind == "batch":  # 4096 reads from each array; payloads of 4, 8 and 16 bytes in turn
        sizes = batching.batched_sizes(c["arrays"], 3)
        b = sum(int(n) * batching.payload_bytes(a) for a, n in enumerate(sizes))
        b += sum(2 * 4096 * batching.payload_bytes(a) for a in range(c["arrays"]))
        b += 2 * 9.3 * min(16, c["arrays"]) * float(sizes.mean())
    elif kind == "serve":
        mean = (c["most"] - 1) / math.log(c["most"])
        flats = min(16, -(-c["arrays"] // max(1, c["arrays"] // c["retire"])))
        b = c["arrays"] * (mean * E + 2 * 4096 * E) + flats * 2 * mean * E
    else:                  # records in, parents read and children written per generation, flatten, passes
        n0, G = c["n0"], c["generations"]
        b = 2 * 16 * n0 + sum(2 * 16 * n0 * 2 ** k for k in range(G))
        b += (2 * 16 + c["passes"] * (16 + 4)) * n0 * 2 ** G
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """Whole numbers and copied bits only: equal or wrong, nothing to be off by."""
    return None
