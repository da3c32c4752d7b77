"""Partition consumer and staged scatter where they can go wrong: bucket counts
on both sides of every flush rule, jobs of different bucket counts in one
launch, tables from one key to overfull, keys that share a home slot.  Results
and filters are integers and must equal the oracle's (or numpy's) exactly."""
import numpy as np
import pytest

import synth
import paper_1712_03254_gb300 as kc

pytestmark = pytest.mark.gpu

M1, M2, GOLD = np.uint64(0xBF58476D1CE4E5B9), np.uint64(0x94D049BB133111EB), np.uint64(0x9E3779B97F4A7C15)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kc.lib()


def _same(c, o):
    keys, counts = c.dump()
    ok, oc = o.result()
    assert np.array_equal(keys, ok)
    assert np.array_equal(counts, oc)
    assert np.array_equal(c.export_bloom(), o.bloom())


@pytest.mark.parametrize("part_bits", [1, 2, 3, 4, 5, 6, 7, 9, 10, 11, 12])
def test_bucket_counts(oracle_mod, part_bits):
    """Every group size of the scatter's flush (a warp, half a warp, ..., one
    thread per bucket) and both stage depths' row strides."""
    w = synth.tiny(scale=0.3)
    w.bloom_bits = 1 << 20
    o = oracle_mod.count(w)
    c = kc.KmerCounter(w.k, 1, w.bloom_bits, w.n_hashes, w.min_count, strategy="partitioned", part_bits=part_bits)
    c.add_readset(0, w.samples[0])
    c.finalize()
    _same(c, o)
    st = c.stats()
    assert st["result_keys"] <= st["table_keys"] <= st["candidates"] <= st["windows"] == o.windows
    c.close()


def test_batch_of_different_bucket_counts(oracle_mod):
    """One batched ingest over jobs of 1024, 2048 and 4096 buckets: each item's
    stages fit the launch's shared memory (2048 buckets take the most)."""
    counters, oracles = [], []
    for i, pb in enumerate((12, 11, 10, 3, 12)):
        g = synth.genome(900 + i, 60_000)
        rs = synth.reads(900 + i, g, 6_000, 60, 160, 0.01, 0.001)
        w = synth.Workload(f"job{i}", [rs], (31, 25)[i % 2], 1 << 20, 4, 2)
        c = kc.KmerCounter(w.k, 1, w.bloom_bits, 4, 2, strategy="partitioned", part_bits=pb, batched_ingest=True)
        c.add_readset(0, rs)
        counters.append(c)
        oracles.append(oracle_mod.count(w))
    b = kc.KcBatch()
    b.ingest(counters)
    b.finalize(counters)
    for c, o in zip(counters, oracles):
        _same(c, o)


def _mixer(x):
    with np.errstate(over="ignore"):
        z = x + GOLD
        z = (z ^ (z >> np.uint64(30))) * M1
        z = (z ^ (z >> np.uint64(27))) * M2
        return z ^ (z >> np.uint64(31))


def _canonical_31mers(rng, n):
    """n distinct canonical 31-mers as (codes uint8[n, 31], keys uint64[n])."""
    codes = rng.integers(0, 4, (n, 31), dtype=np.uint8)
    fwd = np.zeros(n, np.uint64)
    rev = np.zeros(n, np.uint64)
    for i in range(31):
        fwd = (fwd << np.uint64(2)) | codes[:, i].astype(np.uint64)
        rev |= (np.uint64(3) - codes[:, i].astype(np.uint64)) << np.uint64(2 * i)
    keys, at = np.unique(np.minimum(fwd, rev), return_index=True)
    return codes[at], keys


def _count(codes, keys, repeats, samples, min_count, **kw):
    """Key i occurs repeats[s][i] times in sample s; the counter's result against them."""
    c = kc.KmerCounter(31, samples, 1 << 20, 4, min_count, strategy="partitioned", **kw)
    for s in range(samples):
        rows = np.repeat(np.arange(len(keys)), repeats[s])
        np.random.default_rng(5 + s).shuffle(rows)
        ascii = np.frombuffer(b"ACGT", np.uint8)[codes[rows]].reshape(-1)
        c.add_readset(s, synth.ReadSet(ascii, np.arange(len(rows) + 1, dtype=np.uint64) * np.uint64(31)))
    c.finalize()
    got_k, got_c = c.dump()
    total = np.sum(repeats[:samples], axis=0)
    keep = total >= min_count
    assert np.array_equal(got_k, keys[keep])
    assert np.array_equal(got_c, np.stack([repeats[s][keep] for s in range(samples)], 1).astype(np.uint32))
    st = c.stats()
    c.close()
    return st


@pytest.mark.parametrize("samples,min_count", [(1, 1), (1, 2), (2, 2), (2, 3)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 700, 1000, 1024, 1025, 2100])
def test_table_from_one_key_to_overfull(n, samples, min_count):
    """n distinct keys in one partition of a 1024-slot table: rows, queue and
    emission at their edges, then a table that fills up and splits."""
    rng = np.random.default_rng(n)
    codes, keys = _canonical_31mers(rng, 3 * n + 64)
    own = (_mixer(keys) >> np.uint64(63)) == 0  # partition 0 of two
    codes, keys = codes[own][:n], keys[own][:n]
    assert len(keys) == n
    repeats = [rng.integers(0, 4, n) for _ in range(2)]
    repeats[0][:: max(1, n // 3)] += 40  # some keys far above the others
    st = _count(codes, keys, repeats, samples, min_count, part_bits=1, smem_table_log2=10)
    assert st["fallback_partitions"] == 0
    distinct = np.count_nonzero(np.sum(repeats[:samples], axis=0))
    if distinct <= 800:  # at most 0.78 full: 64 probes fail with probability under 800 * 0.78^64 = 1e-4
        assert st["split_partitions"] == 0
    if distinct > 1024:
        assert st["split_partitions"] == 1


@pytest.mark.parametrize("n_same", [2, 33, 64, 66, 90])
def test_keys_of_one_home_slot(n_same):
    """Keys whose hashes end in the same bits as the table's last slot: the probes
    wrap round, and past the probe limit (64, or 65 where the pairs of probes
    begin at an odd one) the partition splits."""
    rng = np.random.default_rng(n_same)
    codes, keys = _canonical_31mers(rng, 400_000)
    h = _mixer(keys)
    own = ((h >> np.uint64(63)) == 0) & ((h & np.uint64(1023)) == 1023)
    codes, keys = codes[own][:n_same], keys[own][:n_same]
    assert len(keys) == n_same
    repeats = [rng.integers(1, 5, n_same), rng.integers(1, 5, n_same)]
    st = _count(codes, keys, repeats, 2, 2, part_bits=1, smem_table_log2=10)
    assert st["fallback_partitions"] == 0
    assert (st["split_partitions"] > 0) == (n_same > 64)


def test_blocks_kept_between_jobs(oracle_mod):
    """Two handles in turn, each reset between jobs of very different sizes, one
    and two kc_add_reads calls, host and device reads: blocks kept for the next
    job never carry anything over."""
    import torch

    g = synth.genome(71, 200_000)
    sets = [synth.reads(71 + n, g, n, 80, 180, 0.01, 0.001) for n in (20_000, 1_500, 30_000, 200, 24_000)]
    oracles = {}
    for k in (31, 25):
        for i, rs in enumerate(sets):
            oracles[k, i] = oracle_mod.count(synth.Workload("job", [rs], k, 1 << 22, 4, 2))
    handles = {k: kc.KmerCounter(k, 1, 1 << 22, 4, 2, strategy="partitioned") for k in (31, 25)}
    for i, rs in enumerate(sets):
        for k, c in handles.items():
            c.reset()
            parts = [rs] if i % 2 == 0 else [rs.slice(0, rs.n_reads // 2), rs.slice(rs.n_reads // 2, rs.n_reads)]
            for p in parts:
                packed, mask = kc.pack_ascii(p.ascii)
                arrays = [packed, np.ascontiguousarray(p.offsets, dtype=np.uint64), mask]
                if k == 25:
                    arrays = [torch.from_numpy(a.view(np.int64)).cuda() for a in arrays]
                    torch.cuda.synchronize()
                c.add_reads(0, *arrays)
            c.finalize()
            _same(c, oracles[k, i])
    for c in handles.values():
        c.close()


def test_sort_buckets_at_both_ends_of_the_key_space():
    """150,000 keys (even-share sort buckets), thousands of them at the very top and
    bottom of the canonical keys: ascending, each with its own count."""
    rng = np.random.default_rng(8)
    codes, _ = _canonical_31mers(rng, 150_000)
    top = rng.integers(0, 4, (3000, 31), dtype=np.uint8)
    top[:, :14], top[:, 17:] = 3, 0  # T...T xyz A...A: both orientations near the top
    low = rng.integers(0, 4, (3000, 31), dtype=np.uint8)
    low[:, :24] = 0
    codes = np.concatenate([codes, top, low])
    w = np.uint64(2)
    fwd = np.zeros(len(codes), np.uint64)
    rev = np.zeros(len(codes), np.uint64)
    for i in range(31):
        fwd = (fwd << w) | codes[:, i].astype(np.uint64)
        rev |= (np.uint64(3) - codes[:, i].astype(np.uint64)) << np.uint64(2 * i)
    keys, at = np.unique(np.minimum(fwd, rev), return_index=True)
    repeats = [rng.integers(1, 4, len(keys))]
    _count(codes[at], keys, repeats, 1, 1)


@pytest.mark.parametrize("k", [31, 17, 4])
@pytest.mark.parametrize("units", [1, 2, 152 * 128, 152 * 128 + 1, 152 * 256, 152 * 512, 152 * 512 + 1])
def test_units_in_parts(oracle_mod, k, units):
    """Reads of so many 64-base units that each CTA's share lies at and above the
    bounds where its lanes take an eighth, a quarter, a half of a unit or all of it."""
    rng = np.random.default_rng(units)
    genome = rng.integers(0, 4, 30_000, dtype=np.uint8)
    n = units * 64 - 21
    lengths = rng.integers(1, 200, n // 60 + 2)
    offsets = np.concatenate([[0], np.minimum(np.cumsum(lengths), n)]).astype(np.uint64)
    offsets = offsets[: int(np.searchsorted(offsets, n)) + 1]
    offsets[-1] = n
    starts = rng.integers(0, len(genome) - 6500, len(offsets) - 1)
    codes = np.concatenate([genome[a : a + int(e - b)] for a, b, e in zip(starts, offsets[:-1], offsets[1:])])
    ascii = np.frombuffer(b"ACGT", np.uint8)[codes].copy()
    ascii[rng.integers(0, n, n // 500 + 1)] = ord("N")
    w = synth.Workload("parts", [synth.ReadSet(ascii, offsets)], k, 1 << 16, 4, 2)
    o = oracle_mod.count(w)
    c = kc.KmerCounter(k, 1, 1 << 16, 4, 2, strategy="partitioned", part_bits=6)
    c.add_readset(0, w.samples[0])
    c.finalize()
    _same(c, o)
    assert c.stats()["windows"] == o.windows
    c.close()


@pytest.mark.parametrize("samples", [1, 2])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 40001])
def test_dump_into_device_arrays(n, samples):
    """Device arrays on and off 16-byte boundaries get what host arrays get, and
    nothing is written behind them."""
    import torch

    rng = np.random.default_rng(n)
    codes, _ = _canonical_31mers(rng, n)
    c = kc.KmerCounter(31, samples, 1 << 16, 4, 1, strategy="partitioned")
    for s in range(samples):
        rows = np.repeat(np.arange(n), rng.integers(1, 4, n))
        ascii = np.frombuffer(b"ACGT", np.uint8)[codes[rows]].reshape(-1)
        c.add_readset(s, synth.ReadSet(ascii, np.arange(len(rows) + 1, dtype=np.uint64) * np.uint64(31)))
    c.finalize()
    keys, counts = c.dump()
    assert len(keys) == n
    for key_at, count_at in ((0, 0), (1, 0), (0, 1), (2, 3), (1, 2)):
        dk = torch.full((n + 4,), -1, dtype=torch.int64, device="cuda")
        dc = torch.full((n * samples + 4,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        c.dump(dk[key_at : key_at + n], dc[count_at : count_at + n * samples])
        dk, dc = dk.cpu().numpy(), dc.cpu().numpy()
        assert np.array_equal(dk[key_at : key_at + n].view(np.uint64), keys)
        assert np.array_equal(dc[count_at : count_at + n * samples].view(np.uint32), counts.reshape(-1))
        assert np.all(np.delete(dk, np.s_[key_at : key_at + n]) == -1)
        assert np.all(np.delete(dc, np.s_[count_at : count_at + n * samples]) == -1)
    c.close()


@pytest.mark.parametrize("sizes", [[32768], [32768, 1], [1, 32768], [31 * 32] * 32 + [1], [32768] * 33 + [40]])
def test_sort_starts_over_several_tiles(sizes):
    """Batches whose sort buckets (sizes / 32 each, at least one) fill one tile of 1024
    counters exactly, pass it by one, and take more tiles than one look-back step."""
    rng = np.random.default_rng(len(sizes))
    jobs = []
    for n in sizes:
        codes, keys = _canonical_31mers(rng, n)
        c = kc.KmerCounter(31, 1, 1 << 20, 4, 1, strategy="partitioned")
        ascii = np.frombuffer(b"ACGT", np.uint8)[codes[rng.permutation(n)]].reshape(-1)
        c.add_readset(0, synth.ReadSet(ascii, np.arange(n + 1, dtype=np.uint64) * np.uint64(31)))
        jobs.append((c, keys))
    kc.KcBatch().finalize([c for c, _ in jobs])
    for c, keys in jobs:
        got, counts = c.dump()
        assert np.array_equal(got, keys) and np.all(counts == 1)
        c.close()


@pytest.mark.parametrize("strategy", ["partitioned", "direct"])
@pytest.mark.parametrize("same", [24, 20, 8])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 63, 64, 65, 256, 257])
def test_sort_bucket_of_n_keys(oracle_mod, n, same, strategy):
    """n keys that begin with `same` As: they share the first sort bucket, spread over
    its ranges (8) or all in one (20, where the keys' top 32 bits are equal, and 24)."""
    rng = np.random.default_rng(1000 * same + n)
    codes = rng.integers(0, 4, (4 * n, 31), dtype=np.uint8)
    codes[:, :same], codes[:, 30] = 0, 1  # the reverse complement begins with G: these are the canonical ones
    codes = np.unique(codes, axis=0)
    codes = codes[np.sort(rng.permutation(len(codes))[:n])]
    assert len(codes) == n
    rows = np.repeat(np.arange(n), rng.integers(1, 5, n))
    rng.shuffle(rows)
    ascii = np.frombuffer(b"ACGT", np.uint8)[codes[rows]].reshape(-1)
    rs = synth.ReadSet(ascii, np.arange(len(rows) + 1, dtype=np.uint64) * np.uint64(31))
    w = synth.Workload("bucket", [rs], 31, 1 << 16, 4, 1)
    o = oracle_mod.count(w)
    kw = dict(table_slots=1 << 12) if strategy == "direct" else {}
    c = kc.KmerCounter(31, 1, 1 << 16, 4, 1, strategy=strategy, **kw)
    c.add_readset(0, rs)
    c.finalize()
    assert len(c.dump()[0]) == n
    _same(c, o)
    c.close()


@pytest.mark.parametrize("k", [31, 20])
@pytest.mark.parametrize("part_bits", [13, 14])
@pytest.mark.parametrize("place", ["device", "chunked"])
def test_two_levels_at_once(oracle_mod, k, part_bits, place):
    """13 and 14 partition bits, reads on the device and host reads copied in
    chunks: streams by the first level's bits, with and without overflow (reads
    that are one key nearly all), and a small batch behind a large one."""
    import torch

    g = synth.genome(51, 100_000)
    poly = synth.ReadSet.from_strings(["A" * 150] * 3_000)
    plain = synth.reads(52, g, 32_000, 120, 160, 0.01, 0.001)
    few = synth.reads(53, g, 40, 20, 90, 0.01, 0.001)
    for sets in ([plain, few], [plain, poly, few]):
        both = synth.ReadSet(np.concatenate([r.ascii for r in sets]),
                             np.concatenate([[0], np.cumsum(np.concatenate([np.diff(r.offsets) for r in sets]))]).astype(np.uint64))
        o = oracle_mod.count(synth.Workload("two", [both], k, 1 << 26, 4, 2))
        c = kc.KmerCounter(k, 1, 1 << 26, 4, 2, strategy="partitioned", part_bits=part_bits)
        for rs in sets:
            packed, mask = kc.pack_ascii(rs.ascii)
            arrays = [packed, np.ascontiguousarray(rs.offsets, dtype=np.uint64), mask]
            if place == "device":
                arrays = [torch.from_numpy(a.view(np.int64)).cuda() for a in arrays]
                torch.cuda.synchronize()
            c.add_reads(0, *arrays)
        assert c.stats()["windows"] == o.windows
        c.finalize()
        _same(c, o)
        c.close()


@pytest.mark.parametrize("samples", [1, 2])
def test_candidates_of_equal_patterns(samples):
    """Keys seen once that share a filter word and its two bits, one in each half of the
    word: whatever their order, the first is new to the filter and every other one a
    candidate."""
    bits, hashes = 1 << 12, 2
    rng = np.random.default_rng(12)
    codes, keys = _canonical_31mers(rng, 1_500_000)
    h = _mixer(keys)
    g = _mixer(h)
    word = (h >> np.uint64(58)).astype(np.int64)
    b0, b1 = (g & np.uint64(63)).astype(np.int64), ((g >> np.uint64(6)) & np.uint64(63)).astype(np.int64)
    lo, hi = np.minimum(b0, b1), np.maximum(b0, b1)
    pick = []
    for w in range(64):  # per word its most frequent pattern over both halves
        at = np.flatnonzero((word == w) & (lo < 32) & (hi >= 32))
        pattern = lo[at] * 64 + hi[at]
        best = np.bincount(pattern).argmax()
        pick.append(at[pattern == best][:40])
    rows = np.concatenate(pick)
    assert all(len(p) > 15 for p in pick)
    reads = np.frombuffer(b"ACGT", np.uint8)[codes[rows]]
    for seed in range(40):
        c = kc.KmerCounter(31, samples, bits, hashes, 2, strategy="partitioned", part_bits=1, smem_table_log2=13)
        order = np.random.default_rng(seed).permutation(len(rows))
        for s, part in enumerate(np.array_split(order, samples)):
            c.add_readset(s, synth.ReadSet(reads[part].reshape(-1), np.arange(len(part) + 1, dtype=np.uint64) * np.uint64(31)))
        c.finalize()
        st = c.stats()
        assert st["windows"] == len(rows) and st["split_partitions"] == 0
        assert st["candidates"] == st["table_keys"] == len(rows) - 64
        assert st["result_keys"] == 0
        c.close()


@pytest.mark.parametrize("samples,split_max", [(1, -1), (1, 1), (2, -1), (2, 2)])
def test_split_limit_is_about_repeated_keys(samples, split_max):
    """70,000 keys of one partition, one in twelve of them more than once: the repeated
    ones fit a table of the library's own size, so a limit on the splits (none at all)
    sends nothing to the global tables."""
    rng = np.random.default_rng(70)
    n = 70_000
    codes, keys = _canonical_31mers(rng, 2 * n + 2000)
    own = (_mixer(keys) >> np.uint64(63)) == 0
    codes, keys = codes[own][:n], keys[own][:n]
    assert len(keys) == n
    repeats = [np.ones(n, np.int64), np.zeros(n, np.int64)]
    repeats[samples - 1][::12] += 2
    st = _count(codes, keys, repeats, samples, 2, part_bits=1, split_max=split_max)
    assert st["fallback_partitions"] == 0 and st["split_partitions"] == 1
