"""Device allocations made to fail on the host (kc_test_fail_alloc: no memory is
filled): a call either reports KC_ERR_OOM_DEVICE and works when it is made again,
or gives the result it gives with memory to spare."""
import ctypes

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


@pytest.fixture
def fail_alloc():
    """fail_alloc(skip, fails): of this thread's allocations the `fails` after the next `skip` fail;
    returns how many there were since the last call."""
    f = kc.lib().kc_test_fail_alloc
    f.restype, f.argtypes = ctypes.c_uint64, (ctypes.c_uint64, ctypes.c_uint64)
    yield f
    f(0, 0)


@pytest.mark.parametrize("n", [0, 1])
def test_batch_object_that_cannot_be_made(fail_alloc, n):
    """kc_batch_create reports the failed allocation and returns (its clean-up once
    waited for a lock that the call itself held)."""
    fail_alloc(n, 1)
    with pytest.raises(kc.KcError) as e:
        kc.KcBatch()
    assert e.value.name == "KC_ERR_OOM_DEVICE"
    fail_alloc(0, 0)
    kc.KcBatch()


def _device(rs):
    import torch

    packed, mask = kc.pack_ascii(rs.ascii)
    arrays = [packed, np.ascontiguousarray(rs.offsets, dtype=np.uint64), mask]
    arrays = [torch.from_numpy(a.view(np.int64)).cuda() for a in arrays]
    torch.cuda.synchronize()
    return arrays


def _expect(o):
    return (*o.result(), o.bloom())


def _same(c, want):
    for x, y in zip((*c.dump(), c.export_bloom()), want):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("how", ["alone", "batch", "batched_ingest"])
def test_finalize_fails_and_is_made_again(oracle_mod, fail_alloc, how):
    """Each allocation of a finalize in turn fails, and all after it, while the handle's
    grouping may still run; another handle's job then takes memory at once, and the
    first one's finalize is made again: both results are the oracle's.  (The reads are
    too many for the finalize to fall back on spilling, and the handle holds blocks from
    earlier jobs, so the survivors' block is the grouping's scratch.)"""
    sets, want = [], []
    for i in range(2):
        g = synth.genome(300 + i, 200_000)
        sets.append(synth.reads(310 + i, g, 40_000, 140, 150, 0.005, 0.0005))
        want.append(_expect(oracle_mod.count(synth.Workload("job", [sets[i]], 31, 1 << 24, 4, 2))))
    dev = [_device(rs) for rs in sets]

    def handle():
        return kc.KmerCounter(31, 1, 1 << 24, 4, 2, strategy="partitioned", batched_ingest=how == "batched_ingest")

    b = handle()
    batch = kc.KcBatch()

    def finalize(c):
        c.finalize() if how == "alone" else batch.finalize([c])

    failed = 0
    for kept in (False, True):  # a handle's first job (result arrays to be made), and its later ones
        for n in range(100):
            if n == 0 or not kept:
                a = handle()
            for _ in range(2 if kept and n == 0 else 0):
                a.add_reads(0, *dev[0])
                finalize(a)
                a.reset()
            a.add_reads(0, *dev[0])
            fail_alloc(n, 1 << 40)
            try:
                finalize(a)
                done = True
            except kc.KcError as e:
                assert e.name == "KC_ERR_OOM_DEVICE"
                done = False
            tried = fail_alloc(0, 0)
            b.reset()
            b.add_reads(0, *dev[1])
            finalize(b)
            if not done:
                failed += 1
                finalize(a)
            _same(a, want[0])
            _same(b, want[1])
            if done and tried <= n:  # every allocation has had its turn
                break
            if kept:
                a.reset()
            else:
                a.close()
        else:
            raise AssertionError("a finalize of more than 100 allocations")
    assert failed > 0
    a.close()
    b.close()


def _keep_blocks(c, arrays):
    """Two jobs and a reset: the handle keeps blocks for its next job."""
    for _ in range(2):
        c.reset()
        c.add_reads(0, *arrays)
        c.finalize()
    c.reset()


def test_any_allocation_may_take_what_idle_handles_keep(oracle_mod, fail_alloc):
    """Each allocation of a handle's life in turn fails once while another handle keeps
    blocks idle: the blocks are given back and the call goes on, result unchanged."""
    g = synth.genome(330, 60_000)
    normal = synth.reads(331, g, 8_000, 90, 120, 0.005, 0.0005)
    tumour = synth.reads(332, synth.mutate(333, g, 0.01, 0.0), 8_000, 90, 120, 0.005, 0.0005)
    o = oracle_mod.count(synth.Workload("job", [normal, tumour], 31, 1 << 22, 4, 2))
    want = _expect(o)
    arrays = [_device(normal), _device(tumour)]
    packed, mask = kc.pack_ascii(tumour.ascii)
    keeper_reads = _device(synth.reads(334, g, 30_000, 90, 120, 0.005, 0.0005))
    keeper = kc.KmerCounter(31, 1, 1 << 22, 4, 2, strategy="partitioned")

    def life(strategy):
        c = kc.KmerCounter(31, 2, 1 << 22, 4, 2, strategy=strategy)
        for s, a in enumerate(arrays):
            c.add_reads(s, *a)
        c.finalize()
        _same(c, want)
        out = [c.export_items(), c.spectrum(15), c.export_stems()]
        c.filter_select(tumor=1, min_tumor=3, max_normal=0)
        out += [*c.filter_keys(), *c.filter_reads(packed, tumour.offsets, mask)]
        c.close()
        return out

    for strategy in ("partitioned", "direct"):
        first = life(strategy)
        for n in range(200):
            _keep_blocks(keeper, keeper_reads)
            kept = keeper.stats()["device_bytes"]
            fail_alloc(n, 1)
            again = life(strategy)
            tried = fail_alloc(0, 0)
            for x, y in zip(first, again):
                assert np.array_equal(x, y)
            if tried <= n:
                break
            assert keeper.stats()["device_bytes"] <= kept - (1 << 20)
        assert 10 < n < 199
    keeper.close()


def test_blocks_taken_back_from_a_busy_handle(oracle_mod, fail_alloc):
    """A handle works job after job on one thread while another thread's allocations
    fail, each taking back what the first one keeps idle at that moment."""
    import threading

    g = synth.genome(340, 200_000)
    rs = synth.reads(341, g, 40_000, 90, 120, 0.005, 0.0005)
    want = _expect(oracle_mod.count(synth.Workload("job", [rs], 31, 1 << 22, 4, 2)))
    arrays = _device(rs)
    stop, wrong = threading.Event(), []

    def busy():
        try:
            c = kc.KmerCounter(31, 1, 1 << 22, 4, 2, strategy="partitioned", batched_ingest=True)
            batch = kc.KcBatch()
            jobs = 0
            while not stop.is_set() or jobs < 3:
                c.reset()
                c.add_reads(0, *arrays)
                batch.ingest([c])
                batch.finalize([c])
                _same(c, want)
                jobs += 1
            c.close()
        except BaseException as e:  # noqa: BLE001 -- reported by the test's own thread
            wrong.append(e)

    t = threading.Thread(target=busy)
    t.start()
    c = kc.KmerCounter(31, 1, 1 << 22, 4, 2, strategy="partitioned")
    for n in range(120):
        c.reset()
        fail_alloc(n % 12, 1)
        try:
            c.add_reads(0, *arrays)
            c.finalize()
            _same(c, want)
        except kc.KcError as e:
            assert e.name == "KC_ERR_OOM_DEVICE"  # nothing was idle at that moment
        fail_alloc(0, 0)
    stop.set()
    t.join()
    assert not wrong, wrong
    c.close()


def _take_back_idle_blocks(fail_alloc):
    """No handle keeps blocks afterwards (a failed allocation takes them back)."""
    fail_alloc(0, 1)
    try:
        kc.KcBatch()
    except kc.KcError:
        pass
    fail_alloc(0, 0)


@pytest.mark.parametrize("call", ["add_reads", "finalize"])
def test_small_job_without_room(oracle_mod, fail_alloc, call):
    """A small job asks for memory without looking whether there is room.  Where there is
    none, its reads are kept and its result spilled: result, filter and counts are those
    of the job that had room, fallback partitions counted once."""
    g = synth.genome(350, 20_000)
    rs = synth.reads(351, g, 6_000, 90, 120, 0.005, 0.0005)
    o = oracle_mod.count(synth.Workload("job", [rs], 31, 1 << 20, 4, 1))
    want = _expect(o)
    arrays = _device(rs)

    def handle():  # every partition too large for its table: global tables
        return kc.KmerCounter(31, 1, 1 << 20, 4, 1, strategy="partitioned", part_bits=2, smem_table_log2=10, split_max=-1)

    c = handle()
    c.add_reads(0, *arrays)
    c.finalize()
    plain = c.stats()
    assert plain["fallback_partitions"] == 4 and plain["candidates"] == o.windows
    c.close()
    spilled = deferred = again = 0
    for n in range(100):
        _take_back_idle_blocks(fail_alloc)
        c = handle()
        for step in ("add_reads", "finalize"):
            def go():
                c.add_reads(0, *arrays) if step == "add_reads" else c.finalize()

            if step == call:
                fail_alloc(n, 1)
            try:
                go()
            except kc.KcError as e:
                assert e.name == "KC_ERR_OOM_DEVICE"
                go()
                again += 1
            if step == call:
                tried = fail_alloc(0, 0)
        st = c.stats()
        for name in ("windows", "candidates", "table_keys", "result_keys", "fallback_partitions", "split_partitions"):
            assert st[name] == plain[name], name
        spilled += st["spilled_bytes"] > 0
        deferred += st["deferred_batches"]
        _same(c, want)
        c.close()
        if tried <= n:
            break
    assert deferred > 0 if call == "add_reads" else spilled > 0


@pytest.mark.parametrize("chain", [False, True])
def test_direct_finalize_made_again(oracle_mod, fail_alloc, chain):
    """The direct strategy counts the reads into its table before the allocations of its
    finalize: a finalize made again does not count them twice, nor where reads are added
    in between."""
    g = synth.genome(360, 30_000)
    rs = synth.reads(361, g, 6_000, 90, 120, 0.005, 0.0005)
    want = _expect(oracle_mod.count(synth.Workload("job", [rs], 31, 1 << 20, 4, 2)))
    arrays, halves = _device(rs), [_device(rs.slice(0, 2_500)), _device(rs.slice(2_500, 6_000))]
    c = kc.KmerCounter(31, 1, 1 << 20, 4, 2, strategy="direct", table_slots=1 << 20, prune_chain=chain)
    again = 0
    for n in range(100):
        _take_back_idle_blocks(fail_alloc)
        c.reset()
        c.add_reads(0, *arrays)
        fail_alloc(n, 1)
        try:
            c.finalize()
        except kc.KcError as e:
            assert e.name == "KC_ERR_OOM_DEVICE"
            c.finalize()
            again += 1
        tried = fail_alloc(0, 0)
        _same(c, want)
        if tried <= n:
            break
        c.reset()
        c.add_reads(0, *halves[0])
        fail_alloc(0, 1 << 40)
        with pytest.raises(kc.KcError):
            c.finalize()
        fail_alloc(0, 0)
        c.add_reads(0, *halves[1])
        c.finalize()
        _same(c, want)
    assert again > 0
    c.close()


@pytest.mark.parametrize("place", ["device", "host"])
def test_failed_calls_keep_no_memory(fail_alloc, place):
    """Many kc_add_reads calls that fail in every place of a two-level grouping, and many
    failed sorts, leave the device's free memory where it was."""
    import torch

    g = synth.genome(370, 300_000)
    rs = synth.reads(371, g, 120_000, 150, 150, 0.005, 0.0005)
    packed, mask = kc.pack_ascii(rs.ascii)
    arrays = _device(rs) if place == "device" else [packed, rs.offsets.astype(np.uint64), mask]
    c = kc.KmerCounter(31, 1, 1 << 28, 4, 2, strategy="partitioned", part_bits=15)
    d = kc.KmerCounter(31, 1, 1 << 24, 4, 1, strategy="direct", table_slots=1 << 23)

    def failing(rounds):
        for n in range(14):
            for _ in range(rounds):
                c.reset()
                fail_alloc(n, 1 << 40)
                try:
                    c.add_reads(0, *arrays)
                except kc.KcError as e:
                    assert e.name == "KC_ERR_OOM_DEVICE"
                fail_alloc(0, 0)
        d.reset()
        d.add_reads(0, *arrays)
        for n in range(10):
            for _ in range(rounds):
                fail_alloc(n, 1 << 40)
                try:
                    d.finalize()
                except kc.KcError as e:
                    assert e.name == "KC_ERR_OOM_DEVICE"
                fail_alloc(0, 0)
        torch.cuda.synchronize()

    c.add_reads(0, *arrays)
    c.finalize()
    failing(1)
    before = torch.cuda.mem_get_info()[0]
    failing(8)
    assert torch.cuda.mem_get_info()[0] > before - (1 << 29)
    c.close()
    d.close()


def test_kept_reads_whose_finalize_fails(oracle_mod, fail_alloc):
    """A job whose reads were kept for want of room, each partition of which goes to a
    global table: every allocation of its finalize fails in turn, and the finalize made
    again after another handle's job gives the oracle's result."""
    g = synth.genome(380, 60_000)
    rs = synth.reads(381, g, 20_000, 90, 120, 0.005, 0.0005)
    other = synth.reads(382, g, 30_000, 90, 120, 0.005, 0.0005)
    want = _expect(oracle_mod.count(synth.Workload("job", [rs], 31, 1 << 20, 4, 2)))
    want_other = _expect(oracle_mod.count(synth.Workload("other", [other], 31, 1 << 22, 4, 2)))
    arrays, other_arrays = _device(rs), _device(other)
    d = kc.KmerCounter(31, 1, 1 << 22, 4, 2, strategy="partitioned")
    failed = 0
    for n in range(0, 400, 7):
        c = kc.KmerCounter(31, 1, 1 << 20, 4, 2, strategy="partitioned", part_bits=2, smem_table_log2=10, split_max=-1,
                           device_budget=(1 << 17) + (8 << 20))
        c.add_reads(0, *arrays)
        assert c.stats()["deferred_batches"] == 1
        _take_back_idle_blocks(fail_alloc)
        fail_alloc(n, 1 << 40)
        try:
            c.finalize()
            done = True
        except kc.KcError as e:
            assert e.name == "KC_ERR_OOM_DEVICE"
            done = False
        tried = fail_alloc(0, 0)
        d.reset()
        d.add_reads(0, *other_arrays)
        d.finalize()
        if not done:
            failed += 1
            c.finalize()
        _same(c, want)
        _same(d, want_other)
        assert c.stats()["fallback_partitions"] > 0
        c.close()
        if tried <= n:
            break
    assert failed > 0
    d.close()


def test_idle_blocks_of_a_stream_in_a_capture(fail_alloc):
    """A handle on a caller's stream keeps blocks while the caller captures that stream: an
    allocation that fails on another thread leaves the blocks and the capture alone."""
    import threading

    import torch

    g = synth.genome(390, 60_000)
    arrays = _device(synth.reads(391, g, 30_000, 90, 120, 0.005, 0.0005))
    stream = torch.cuda.Stream()
    c = kc.KmerCounter(31, 1, 1 << 22, 4, 2, strategy="partitioned", stream=stream.cuda_stream)
    _take_back_idle_blocks(fail_alloc)
    _keep_blocks(c, arrays)
    kept = c.stats()["device_bytes"]
    x = torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    seen = []

    def other():
        fail_alloc(0, 1)
        try:
            kc.KcBatch()
        except kc.KcError as e:
            seen.append(e.name)
        fail_alloc(0, 0)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        x.add_(1)
        t = threading.Thread(target=other)
        t.start()
        t.join()
        x.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert seen == ["KC_ERR_OOM_DEVICE"] and c.stats()["device_bytes"] == kept
    assert float(x.sum()) == 128.0
    c.add_reads(0, *arrays)
    c.finalize()
    assert c.result_size() > 0
    c.close()
