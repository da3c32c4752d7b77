"""The work a user of this library has it do, as cases that can be timed.

Each case is one job, or one batch of jobs, through the package's public entry
points, on seeded synthetic reads with the shapes of the repository's own
workloads (``synth``: tiny, mid, paired, ooc, served) and of its tests:

* ``count``       reads in, sorted keys and counts out (``KmerCounter``): one
                  or two samples, reads on the device or in host memory, a
                  handle kept from job to job or made for one job, with or
                  without the filter's words, spilled or not, the two-filter
                  Prune chain
* ``batch``       several small jobs grouped and finalized together (``KcBatch``)
* ``rescan``      the Filter unit: select the tumour's k-mers of a finished
                  joint count, then look every read of both samples up
* ``downstream``  a joint count and what is exported from it: 16-byte items,
                  the count spectrum, the stem table
"""
import math

import numpy as np
import torch

import paper_1712_03254_gb300 as kc

DEV = "cuda"
BASE = {
    "kind": "count", "k": 31, "samples": 1, "genome": 100_000, "reads": 20_000, "len_min": 100, "len_max": 100,
    "sub": 0.005, "n_rate": 0.0005, "bloom_log2": 24, "hashes": 4, "min_count": 2, "where": "device", "fresh": False,
    "words": False, "chain": False, "spill": 0, "jobs": 1,
}


def _case(**kw):
    return {**BASE, **kw}


def _served_log2(genome, windows, k, sub):
    """Filter bits of a served job: 8 per expected distinct k-mer (as synth.served_bloom_bits)."""
    expected = genome + windows * (1.0 - (1.0 - sub) ** k)
    return max(12, math.ceil(math.log2(max(1.0, 8.0 * expected))))


def _served(genome, reads, k, **kw):
    windows = reads * max(1, 175 - k + 1)
    return _case(genome=genome, reads=reads, len_min=100, len_max=250, k=k,
                 bloom_log2=_served_log2(genome, windows, k, 0.005), **kw)


def listed():
    return [
        # the smallest job, again and again on one handle, its filter read out as a checkpoint does: latency, launches
        _case(name="tiny", sub=0.01, n_rate=0.001, words=True),
        # a single small job of a program that counts once: pageable arrays in, numpy arrays out, handle made and closed
        _served(1_000_000, 10_000, 25, where="host", fresh=True) | {"name": "one_small_job"},
        # the benchmark's workload: 30x coverage, reads and result on the device
        _case(name="mid", genome=5_000_000, reads=1_000_000, len_min=150, len_max=150, bloom_log2=30),
        # the same from pinned host buffers into pinned host buffers, as reads come from a loader
        _case(name="mid_host", genome=5_000_000, reads=1_000_000, len_min=150, len_max=150, bloom_log2=30, where="pinned"),
        # a large served job: ragged reads, k = 25, filter of about 8 bits per distinct k-mer
        _served(12_000_000, 1_200_000, 25) | {"name": "served_large"},
        # a served job of low coverage, where most k-mers are seen once and the filter keeps them out of the table
        _served(20_000_000, 200_000, 31) | {"name": "served_sparse"},
        # every k-mer kept (min_count 1), a shorter k, fewer hashes: a k-mer spectrum
        _case(name="keep_all", k=21, genome=3_000_000, reads=300_000, len_min=150, len_max=150, bloom_log2=28, hashes=2,
              min_count=1),
        # normal and tumour counted into one joint table, a filter that takes two grouping levels
        _case(name="joint", samples=2, genome=10_000_000, reads=2_000_000, len_min=150, len_max=150, bloom_log2=32),
        # what follows a joint count: items, spectrum, stem table
        _case(name="downstream", kind="downstream", samples=2, genome=1_000_000, reads=200_000, len_min=150, len_max=150,
              bloom_log2=28),
        # the Filter unit on a finished joint count: selection, then every read of both samples
        _case(name="rescan", kind="rescan", samples=2, genome=5_000_000, reads=600_000, len_min=150, len_max=150,
              bloom_log2=30),
        # a burst of served jobs finalized together
        _case(name="batch", kind="batch", jobs=12, genome=3_000_000, reads=60_000, len_min=100, len_max=250, where="pinned"),
        # the paper's two-filter chain
        _case(name="prune_chain", genome=1_000_000, reads=200_000, len_min=150, len_max=150, bloom_log2=28, chain=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count"] * 6 + ["batch", "rescan", "downstream", "chain"])
    k = rng.choice([31, 31, 31, 25, 25, 27, 29, 21, 30])
    length = rng.choice([100, 150, 150, 0, 0])  # 0: ragged, 100..250
    reads = _log(rng, 5_000, 1_500_000)
    genome = max(50_000, int(reads * 150 / rng.uniform(4, 60)))
    lo, hi = (length, length) if length else (100, 250)
    windows = reads * ((lo + hi) // 2 - k + 1)
    log2 = _served_log2(genome, windows, k, 0.005)
    c = _case(k=k, genome=genome, reads=reads, len_min=lo, len_max=hi, bloom_log2=min(32, log2 + rng.choice([0, 0, 1, 3])),
              sub=rng.choice([0.002, 0.005, 0.01]), n_rate=rng.choice([0.0, 0.0005, 0.001]), hashes=rng.choice([4, 4, 4, 3, 6]),
              min_count=rng.choice([2, 2, 2, 3, 1]), where=rng.choice(["device", "device", "pinned", "host"]),
              samples=rng.choice([1, 1, 2]), fresh=rng.random() < 0.2, words=rng.random() < 0.3)
    if kind == "batch":
        n = _log(rng, 10_000, 200_000)
        c.update(kind="batch", jobs=rng.randint(2, 16), reads=n, genome=max(50_000, n * 150 // rng.randint(4, 40)), samples=1,
                 fresh=False, words=False, where="pinned")
    elif kind in ("rescan", "downstream"):
        n = _log(rng, 20_000, 800_000)
        c.update(kind=kind, samples=2, reads=n, genome=max(50_000, n * 150 // rng.randint(10, 40)), min_count=2, where="device",
                 fresh=False, words=False, k=rng.choice([31, 31, 25, 30]))
    elif kind == "chain":
        n = _log(rng, 10_000, 300_000)
        c.update(chain=True, samples=1, reads=n, genome=max(50_000, n * 150 // rng.randint(10, 40)), min_count=2, words=False)
    elif reads < 400_000 and rng.random() < 0.2:
        c.update(spill=rng.choice([1, 2]), fresh=False)  # results that go out to pinned host memory
    return c


# ---- inputs --------------------------------------------------------------------


def _genome(gen, n):
    return torch.randint(0, 4, (n,), generator=gen, device=DEV, dtype=torch.uint8)


def _mutated(gen, g, rate):
    hit = torch.rand(g.numel(), generator=gen, device=DEV) < rate
    shift = torch.randint(1, 4, (g.numel(),), generator=gen, device=DEV, dtype=torch.uint8)
    return torch.where(hit, (g + shift) & 3, g)


def _pack(codes, unknown):
    """(packed, n_mask) int64 words of 2-bit codes and unknown flags, the first base in the top bits."""
    n = codes.numel()
    s2 = torch.arange(62, -1, -2, device=DEV)
    s1 = torch.arange(63, -1, -1, device=DEV)
    packed = torch.zeros((n + 31) // 32, dtype=torch.int64, device=DEV)
    mask = torch.zeros((n + 63) // 64, dtype=torch.int64, device=DEV)
    step = 1 << 25
    for a in range(0, n, step):
        c, u = codes[a:a + step], unknown[a:a + step]
        pad = -c.numel() % 64
        if pad:
            c, u = torch.nn.functional.pad(c, (0, pad)), torch.nn.functional.pad(u, (0, pad))
        pw = (c.view(-1, 32).to(torch.int64) << s2).sum(1)
        mw = (u.view(-1, 64).to(torch.int64) << s1).sum(1)
        packed[a // 32:a // 32 + pw.numel()] = pw[:packed.numel() - a // 32]
        mask[a // 64:a // 64 + mw.numel()] = mw
    return packed, mask


def _reads(gen, g, n_reads, lo, hi, sub, n_rate):
    """Reads from either strand at uniform places: (codes, unknown flags, offsets)."""
    lens = torch.randint(lo, hi + 1, (n_reads,), generator=gen, device=DEV)
    offsets = torch.zeros(n_reads + 1, dtype=torch.int64, device=DEV)
    offsets[1:] = lens.cumsum(0)
    total = int(offsets[-1])
    start = (torch.rand(n_reads, generator=gen, device=DEV, dtype=torch.float64) * (g.numel() - lens + 1)).long()
    flip = torch.rand(n_reads, generator=gen, device=DEV) < 0.5
    codes = torch.empty(total, dtype=torch.uint8, device=DEV)
    unknown = torch.empty(total, dtype=torch.bool, device=DEV)
    step = 1 << 18
    for r in range(0, n_reads, step):
        ln, e = lens[r:r + step], min(n_reads, r + step)
        a, b = int(offsets[r]), int(offsets[e])
        j = torch.arange(b - a, device=DEV) - torch.repeat_interleave(offsets[r:e] - a, ln)
        f = torch.repeat_interleave(flip[r:e], ln)
        at = torch.repeat_interleave(start[r:e], ln) + torch.where(f, torch.repeat_interleave(ln, ln) - 1 - j, j)
        c = g[at]
        c = torch.where(f, 3 - c, c)
        wrong = torch.rand(b - a, generator=gen, device=DEV) < sub
        shift = torch.randint(1, 4, (b - a,), generator=gen, device=DEV, dtype=torch.uint8)
        codes[a:b] = torch.where(wrong, (c + shift) & 3, c)
        unknown[a:b] = torch.rand(b - a, generator=gen, device=DEV) < n_rate
    return codes, unknown, offsets


def _job_cases(case):
    """The jobs of a case: itself, or a batch's jobs (sizes spread over a factor of eight, k 25 and 31)."""
    if case["kind"] != "batch":
        return [case]
    out = []
    for i in range(case["jobs"]):
        f = 2.0 ** (3.0 * i / max(1, case["jobs"] - 1) - 1.5)
        n, g, k = max(100, int(case["reads"] * f)), max(50_000, int(case["genome"] * f)), (25, 31)[i % 2]
        windows = n * ((case["len_min"] + case["len_max"]) // 2 - k + 1)
        out.append({**case, "reads": n, "genome": g, "k": k, "bloom_log2": _served_log2(g, windows, k, 0.005)})
    return out


def _raw_inputs(case, seed):
    """Per job, per sample: (codes, unknown, offsets) on the device."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed * 1_000_003 + 17)
    jobs = []
    for j in _job_cases(case):
        g = _genome(gen, j["genome"])
        genomes = [g] if j["samples"] == 1 else [g, _mutated(gen, g, 0.001)]
        jobs.append([_reads(gen, x, j["reads"], j["len_min"], j["len_max"], j["sub"], j["n_rate"]) for x in genomes])
    return jobs


def _placed(codes, unknown, offsets, where):
    packed, mask = _pack(codes, unknown)
    arrays = (packed, offsets, mask)
    if where == "pinned":
        return tuple(t.cpu().pin_memory() for t in arrays)
    if where == "host":
        return tuple(t.cpu().numpy().view(np.uint64) for t in arrays)
    return arrays


def _counter(j, **kw):
    return kc.KmerCounter(j["k"], j["samples"], 1 << j["bloom_log2"], j["hashes"], j["min_count"],
                          strategy="direct" if j["chain"] else "auto", prune_chain=j["chain"], spill=j["spill"], **kw)


def prepare(case, seed):
    jobs = _job_cases(case)
    inputs = [[_placed(*s, case["where"]) for s in samples] for samples in _raw_inputs(case, seed)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()  # the library's allocations do not come out of torch's pool
    state = {"case": case, "jobs": jobs, "inputs": inputs}
    if not case["fresh"]:
        state["counters"] = [_counter(j, batched_ingest=case["kind"] == "batch") for j in jobs]
    if case["kind"] == "batch":
        state["batch"] = kc.KcBatch()
    state["results"] = [_room(j) for j in jobs]
    if case["words"]:
        state["words"] = _zeros(case, (1 << case["bloom_log2"]) // 64, np.int64)
    if case["kind"] == "downstream":
        cap = _capacity(case)
        state["items"], state["stems"] = _zeros(case, 2 * cap, np.int64), _zeros(case, 9 * cap, np.int64)
    if case["kind"] == "rescan":  # the finished joint count the selection works on
        c = state["counters"][0]
        _add(c, inputs[0])
        c.finalize()
        cap = _capacity(case)
        state["selected"] = [np.zeros(cap, np.int64), np.zeros((cap, 2), np.int32)]
        state["hits"] = [_zeros(case, case["reads"], np.int32) for _ in inputs[0]]
        state["which"] = [_zeros(case, case["reads"], np.int64) for _ in inputs[0]]
    return state


def _expected_keys(j):
    """Expected keys of a job's result."""
    per = max(0.0, (j["len_min"] + j["len_max"]) / 2 - j["k"] + 1)
    windows = j["samples"] * j["reads"] * per
    good = (1.0 - j["sub"]) ** j["k"] * (1.0 - j["n_rate"]) ** j["k"]
    cover = windows * good / j["genome"]  # expected error-free windows per genome position
    below = math.exp(-cover) * sum(cover ** i / math.factorial(i) for i in range(min(j["min_count"], 8)))
    return j["genome"] * (1.0 - below) + (windows * (1.0 - good) if j["min_count"] == 1 else 0.0)


def _capacity(j):
    """Keys the result arrays are given room for: well above what the job can be expected to keep."""
    return int(2.0 * _expected_keys(j)) + 50_000


def _zeros(case, n, dtype):
    """A result buffer where the case has its arrays: on the device, in pinned memory, or a numpy array."""
    if case["where"] == "host":
        return np.zeros(n, dtype)
    t = torch.int64 if dtype == np.int64 else torch.int32
    return torch.zeros(n, dtype=t, device=DEV) if case["where"] == "device" else torch.zeros(n, dtype=t).pin_memory()


def _room(j):
    return [_zeros(j, _capacity(j), np.int64), _zeros(j, (_capacity(j), j["samples"]), np.int32)]


def _add(c, samples):
    for s, arrays in enumerate(samples):
        c.add_reads(s, *arrays)


def _dump(c, room):
    """The whole result into its buffers (zeros behind it), and how many keys it has."""
    n = c.result_size()
    if n:
        c.dump(*room)
    return [*room, n]


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        for c, samples in zip(state["counters"], state["inputs"]):
            c.reset()
            _add(c, samples)
        state["batch"].ingest(state["counters"])
        state["batch"].finalize(state["counters"])
        return [_dump(c, room) for c, room in zip(state["counters"], state["results"])]
    if case["kind"] == "rescan":
        c = state["counters"][0]
        n = c.filter_select(tumor=1, min_tumor=4, max_normal=0)
        keys, counts = c.filter_keys()
        state["selected"][0][:n], state["selected"][1][:n] = keys, counts
        out = [*state["selected"], n]
        for (packed, offsets, mask), hits, which in zip(state["inputs"][0], state["hits"], state["which"]):
            out += [hits, which, c.filter_reads(packed, offsets, mask, hits=hits, candidates=which)[2]]
        return out
    c = _counter(state["jobs"][0]) if case["fresh"] else state["counters"][0]
    if not case["fresh"]:
        c.reset()
    _add(c, state["inputs"][0])
    c.finalize()
    out = _dump(c, state["results"][0])
    if case["words"]:
        out.append(c.export_bloom(out=state["words"]))
    if case["kind"] == "downstream":
        out += [c.export_items(state["items"]), c.spectrum(63).view(np.int64), c.export_stems(state["stems"])]
    if case["fresh"]:
        c.close()
    return out


def work(case):
    """Compulsory bytes of one pass: the reads at 3 bits a base and their offsets once, the filter written once, the
    expected result written once (and the exports); operations: a few integer ones per window and filter bit."""
    total_bytes, total_ops = 0.0, 0.0
    for j in _job_cases(case):
        length = (j["len_min"] + j["len_max"]) / 2
        windows = j["samples"] * j["reads"] * max(0.0, length - j["k"] + 1)
        keys = _expected_keys(j)
        reads_in = j["samples"] * (j["reads"] * length * 3 / 8 + 8 * (j["reads"] + 1))
        if case["kind"] == "rescan":
            total_bytes += reads_in + 4 * 2 * j["reads"] + 8 * keys  # hits out; the counts read to select
        else:
            total_bytes += reads_in + (1 << j["bloom_log2"]) / 8 + keys * (8 + 4 * j["samples"])
            if case["kind"] == "downstream":
                total_bytes += keys * (16 + 72)
        total_ops += windows * (8 + 2 * j["hashes"])
    return {"bytes": total_bytes, "flops": total_ops}


# ---- what run() returns, from the definition ------------------------------------


def _srl(x, s):
    """Logical right shift of int64 words."""
    return (x >> s) & ((1 << (64 - s)) - 1)


def _i64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _mixer(x):
    z = x + _i64(0x9E3779B97F4A7C15)
    z = (z ^ _srl(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _srl(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _srl(z, 31)


def _canonical(codes, unknown, offsets, k):
    """Canonical keys of all valid windows of the reads."""
    n = codes.numel()
    if n < k:
        return torch.empty(0, dtype=torch.int64, device=DEV)
    m = n - k + 1
    first = torch.zeros(n, dtype=torch.int32, device=DEV)
    inner = offsets[1:-1]
    first[inner[inner < n]] = 1
    bad = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    bad[1:] = unknown.to(torch.int32).cumsum(0)
    brk = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    brk[1:] = first.cumsum(0)
    ok = (bad[k:k + m] == bad[:m]) & (brk[k:k + m] == brk[1:1 + m])
    fwd = torch.zeros(m, dtype=torch.int64, device=DEV)
    rev = torch.zeros(m, dtype=torch.int64, device=DEV)
    for i in range(k):
        c = codes[i:i + m].to(torch.int64)
        fwd = (fwd << 2) | c
        rev |= (3 - c) << (2 * i)
    return torch.minimum(fwd, rev)[ok]


def _exact_job(samples, j, words):
    per = [_canonical(*s, j["k"]) for s in samples]
    keys, inv = torch.unique(torch.cat(per), return_inverse=True)
    counts = torch.zeros((keys.numel(), len(per)), dtype=torch.int64, device=DEV)
    a = 0
    for s, p in enumerate(per):
        counts[:, s] = torch.bincount(inv[a:a + p.numel()], minlength=keys.numel())
        a += p.numel()
    keep = counts.sum(1) >= j["min_count"]
    n, cap = int(keep.sum()), _capacity(j)
    out = [torch.zeros(cap, dtype=torch.int64, device=DEV), torch.zeros((cap, len(per)), dtype=torch.int32, device=DEV), n]
    out[0][:n], out[1][:n] = keys[keep], counts[keep].to(torch.int32)
    if words:
        h = _mixer(keys)
        g = _mixer(h)
        word = _srl(h, 64 - (j["bloom_log2"] - 6))
        bits = torch.zeros(1 << j["bloom_log2"], dtype=torch.bool, device=DEV)
        for i in range(j["hashes"]):
            bits[word * 64 + ((g >> (6 * i)) & 63)] = True
        out.append((bits.view(-1, 64).to(torch.int64) << torch.arange(64, device=DEV)).sum(1))
    return out


def exact(case, seed):
    """Keys, counts and filter words from the definition (plain torch, 64-bit); the exports and the rescan have none."""
    windows = sum(j["samples"] * j["reads"] * (j["len_min"] + j["len_max"]) // 2 for j in _job_cases(case))
    if case["kind"] == "rescan" or windows > 200_000_000 or (case["words"] and case["bloom_log2"] > 30):
        return None
    out = []
    for j, samples in zip(_job_cases(case), _raw_inputs(case, seed)):
        out.append(_exact_job(samples, j, case["words"]))
    if case["kind"] == "batch":
        return out
    return out[0] + ([None, None, None] if case["kind"] == "downstream" else [])
