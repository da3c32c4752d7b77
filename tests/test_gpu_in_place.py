"""Reads given in device memory are read where they are: without the padding of
the library's own copy, at any 8-byte alignment, up to the last base exactly."""
import numpy as np
import pytest

import synth
import paper_1712_03254_gb300 as kc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kc.lib()


def _on_device(a, shift):
    """The array on the device, `shift` words behind a 16-byte boundary, with no word after it."""
    import torch

    t = torch.empty(len(a) + shift, dtype=torch.int64, device="cuda")
    t[shift:] = torch.from_numpy(np.ascontiguousarray(a).view(np.int64))
    return t[shift:]


@pytest.mark.parametrize("k", [5, 16, 17, 25, 31])
@pytest.mark.parametrize("tail", [1, 31, 32, 33, 63, 64])
def test_filter_reads_in_place(oracle_mod, k, tail):
    """Hits of device reads (aligned and not) are those of host reads, and their
    sum is the selected keys' counts; the last unit holds `tail` bases."""
    import torch

    g = synth.genome(41, 3_000 if k > 5 else 120)
    normal = synth.reads(42, g, 400, 60, 100, 0.01, 0.002)
    rs = synth.reads(43, synth.mutate(44, g, 0.02, 0.0), 400, 60, 100, 0.01, 0.002)
    keep = rs.n_reads
    cut = int(rs.offsets[-1]) - (int(rs.offsets[-1]) - tail) % 64  # bases = tail mod 64
    rs = synth.ReadSet(rs.ascii[:cut], np.minimum(rs.offsets, np.uint64(cut)))
    c = kc.KmerCounter(k, 2, 1 << 18, 4, 2)
    c.add_readset(0, normal)
    c.add_readset(1, rs)
    c.finalize()
    n_sel = c.filter_select(tumor=1, min_tumor=2, max_normal=3)
    packed, mask = kc.pack_ascii(rs.ascii)
    want, cand, n = c.filter_reads(packed, rs.offsets, mask)
    if n_sel:
        assert int(want.sum()) == int(c.filter_keys()[1][:, 1].sum())
    assert np.array_equal(cand, np.flatnonzero(want)) and n == len(cand)
    for shift in (0, 1):
        torch.cuda.synchronize()
        args = [_on_device(packed, shift), _on_device(rs.offsets, shift), _on_device(mask, shift)]
        torch.cuda.synchronize()
        hits = torch.full((keep,), -1, dtype=torch.int32, device="cuda")
        which = torch.full((keep,), -1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        _, _, m = c.filter_reads(*args, hits=hits, candidates=which)
        assert m == n
        assert np.array_equal(hits.cpu().numpy(), want.astype(np.int32))
        assert np.array_equal(which[:m].cpu().numpy(), cand.astype(np.int64))
    c.close()


def test_filter_reads_without_bases():
    """Reads that are all empty behind a base offset: no word is read, no hit."""
    c = kc.KmerCounter(5, 2, 1 << 12, 4, 1)
    rs = synth.ReadSet.from_strings(["ACGTTGCA", "ACGTAGCA"])
    c.add_readset(0, rs)
    c.add_readset(1, rs)
    c.finalize()
    c.filter_select(tumor=1, min_tumor=1, max_normal=5)
    offsets = np.full(4, 100, dtype=np.uint64)
    hits, cand, n = c.filter_reads(np.zeros(1, np.uint64), offsets, np.zeros(1, np.uint64))
    assert n == 0 and len(cand) == 0 and not hits.any()
    c.close()


@pytest.mark.parametrize("units", [155648 // 8, 155648 // 8 + 1, 155648 // 4, 155648 // 4 + 1, 155648 // 2,
                                   155648 // 2 + 1, 155648 + 5])
def test_filter_units_in_parts(units):
    """Rescans whose units fill the lanes an eighth, a quarter, half or a whole time, exactly
    and passed by one: the hits of every read are those of the reads scanned in pieces, and add
    up to the selected keys' counts."""
    rng = np.random.default_rng(units)
    genome = rng.integers(0, 4, 20_000, dtype=np.uint8)
    letters = np.frombuffer(b"ACGT", np.uint8)
    n = units * 64 - 13
    bounds = np.append(np.arange(0, n - 300, 150), n).astype(np.uint64)
    starts = rng.integers(0, len(genome) - 500, len(bounds) - 1)
    lengths = np.diff(bounds).astype(np.int64)
    at = np.repeat(starts, lengths) + np.arange(n) - np.repeat(bounds[:-1].astype(np.int64), lengths)
    tumour = synth.ReadSet(letters[genome[at]], bounds)
    normal = synth.ReadSet.from_strings([letters[genome[:15_000]].tobytes().decode()])
    c = kc.KmerCounter(25, 2, 1 << 20, 4, 2)
    c.add_readset(0, normal)
    c.add_readset(1, tumour)
    c.finalize()
    assert c.filter_select(tumor=1, min_tumor=2, max_normal=0) > 0
    hits, _, _ = c.filter_readset(tumour)
    assert int(hits.sum()) == int(c.filter_keys()[1][:, 1].sum())
    pieces = np.array_split(np.arange(tumour.n_reads), 7)
    parts = [c.filter_readset(tumour.slice(int(p[0]), int(p[-1]) + 1))[0] for p in pieces]
    assert np.array_equal(hits, np.concatenate(parts))
    c.close()


@pytest.mark.parametrize("shift", [1, 4, 6])
def test_device_arrays_at_odd_addresses(oracle_mod, shift):
    """Packed words, offsets and N mask in device memory, `shift` bytes behind an 8-byte
    boundary, are copied: the counts are the oracle's, the hits those of host reads."""
    import ctypes

    import torch

    g = synth.genome(45, 5_000)
    rs = synth.reads(46, g, 700, 60, 100, 0.01, 0.002)
    other = synth.reads(47, g, 300, 60, 100, 0.01, 0.002)
    w = synth.Workload("odd", [other, rs], 31, 1 << 18, 4, 2)
    o = oracle_mod.count(w)
    packed, mask = kc.pack_ascii(rs.ascii)
    held = []

    def odd(a):
        raw = np.ascontiguousarray(a).view(np.uint8)
        t = torch.zeros(len(raw) + 16, dtype=torch.uint8, device="cuda")
        assert t.data_ptr() % 8 == 0
        t[shift : shift + len(raw)] = torch.from_numpy(raw.copy())
        held.append(t)
        return ctypes.c_void_p(t.data_ptr() + shift)

    args = [odd(packed), odd(rs.offsets.astype(np.uint64)), odd(mask)]
    torch.cuda.synchronize()
    for strategy in ("partitioned", "direct"):
        c = kc.KmerCounter(31, 2, 1 << 18, 4, 2, strategy=strategy)
        c.add_readset(0, other)
        assert c._L.kc_add_reads(c._h, 1, *args, rs.n_reads) == 0
        c.finalize()
        for x, y in zip(c.dump(), o.result()):
            assert np.array_equal(x, y)
        c.filter_select(tumor=1, min_tumor=2, max_normal=1)
        want, _, n = c.filter_reads(packed, rs.offsets, mask)
        hits, m = np.zeros(rs.n_reads, np.uint32), ctypes.c_uint64()
        assert c._L.kc_filter_reads(c._h, *args, rs.n_reads, hits.ctypes.data_as(ctypes.c_void_p), None, ctypes.byref(m)) == 0
        assert m.value == n > 0 and np.array_equal(hits, want)
        c.close()


@pytest.mark.parametrize("rest", [1, 155648 // 8, 155648 // 8 + 1, 155648 // 4, 155648 // 4 + 1, 155648 // 2,
                                  155648 // 2 + 1])
def test_filter_rest_of_units_in_parts(rest):
    """The same behind a whole round of the lanes (152 CTAs of 1024): a rest whose units are
    taken in eighths, quarters, halves and whole, so that the hit mask is written in bytes,
    in 16 and in 32 bits."""
    import torch

    lanes = torch.cuda.get_device_properties(0).multi_processor_count * 1024
    test_filter_units_in_parts(lanes + rest * lanes // 155648)
