"""Growth of the storage layer on a stream of the library's own, and growth that fails part-way."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_results_equal, assert_state_equal, make_index, results_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc_mod():
    import oracle
    oracle.build()
    return oracle


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    from paper_1601_00159_gb300 import build, load_library
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return load_library()


def host_batch(b):
    import torch
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a.view(np.int64) if a.dtype == np.uint64 else a)).pin_memory()
    return pin(b.ops), pin(b.keys), pin(b.vals), torch.empty((len(b), 2), dtype=torch.int64, pin_memory=True)


def inserts(seed, first, q):
    k = wl.distinct_keys(seed, np.uint64(first) + np.arange(q, dtype=np.uint64))
    return wl.Batch(np.full(q, 1, np.uint8), k, wl.u64_stream(wl.stream_seed(seed, first), 0, q))


@pytest.mark.parametrize("flags", [0, 0x100])
def test_growth_while_the_default_stream_is_busy(orc_mod, flags):
    """The host-buffer call works on streams that the default stream does not hold back. Its growth
    must not leave a clear of the new arrays to the default stream, where it would come after the
    copy of the nodes, with their heights and delete flags."""
    import torch
    n, q = 70_000, 100_000
    keys = wl.distinct_keys(97, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 11, {"test_flags": flags} if flags else None)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 11)
    gone = keys[::14]
    batches = [wl.Batch(np.full(len(gone), 2, np.uint8), gone, gone), inserts(97, 1_000_000, q)]
    searches = np.concatenate([keys, batches[1].keys])
    batches.append(wl.Batch(np.zeros(len(searches), np.uint8), searches, searches))
    cap = idx.info()["storage_capacity"]
    assert n + q > cap
    dev = [host_batch(b) for b in batches]
    idx.execute_host(*dev[0])
    torch.cuda.synchronize()
    for d in dev[1:]:
        torch.cuda._sleep(200_000_000)  # some 100 ms of the default stream
        idx.execute_host(*d)
    torch.cuda.synchronize()
    for i, (b, d) in enumerate(zip(batches, dev)):
        assert_results_equal(results_np(d[3]), orc.execute(b.ops, b.keys, b.vals), f"batch {i}")
    info = assert_state_equal(idx, orc)
    assert info["storage_capacity"] > cap
    idx.close()
    orc.close()


@pytest.mark.parametrize("flags,allocs", [(0, 3), (0x100, 4)])  # storage, look-back words, counts (, write counters)
@pytest.mark.parametrize("skip", [0, 1, 2, 3, 4])
def test_growth_that_fails_part_way(orc_mod, flags, allocs, skip):
    """Whichever of a growth's allocations fails, the batch is refused with the index as it was, and
    the batches after it are right; once all of them succeed, nothing is refused."""
    import paper_1601_00159_gb300 as pkg
    from tests.parity import run_batch
    n, q = 70_000, 60_000
    keys = wl.distinct_keys(98, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 12, {"test_flags": flags} if flags else None)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 12)
    first = inserts(98, 500_000, q)  # the scratch's growth, and nodes up to near the capacity
    assert_results_equal(run_batch(idx, first), orc.execute(first.ops, first.keys, first.vals), "first")
    cap = idx.info()["storage_capacity"]
    assert n + q < cap < n + 2 * q
    batches = [inserts(98, 1_000_000, q), inserts(98, 2_000_000, q // 2), inserts(98, 1_020_000, q)]
    pkg.test_fail_allocations(1, skip)
    try:
        if skip < allocs:
            with pytest.raises(pkg.PiError) as ei:
                run_batch(idx, batches[0])
            assert ei.value.code == pkg.PI_ERR_OOM
            pkg.test_fail_allocations(0)
            assert idx.info()["storage_capacity"] == cap
            assert_state_equal(idx, orc, "after the refused batch")
            fits = wl.Batch(np.full(5000, 2, np.uint8), keys[:5000], keys[:5000])
            assert_results_equal(run_batch(idx, fits), orc.execute(fits.ops, fits.keys, fits.vals), "one that fits")
        for i, b in enumerate(batches):
            assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals), f"batch {i}")
    finally:
        pkg.test_fail_allocations(0)
    info = assert_state_equal(idx, orc, "end")
    assert info["storage_capacity"] > cap
    idx.close()
    orc.close()


@pytest.mark.parametrize("skip", [0, 1, 2, 3])
def test_scratch_growth_that_fails_part_way(orc_mod, skip):
    """A batch that outgrows the scratch, the look-back words and the storage layer at once."""
    import paper_1601_00159_gb300 as pkg
    from tests.parity import run_batch
    n, q = 10_000, 1 << 21
    keys = wl.distinct_keys(99, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 14)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 14)
    small = inserts(99, 500_000, 3000)
    assert_results_equal(run_batch(idx, small), orc.execute(small.ops, small.keys, small.vals), "small")
    big = wl.Batch(np.zeros(q, np.uint8), np.resize(keys, q), np.resize(keys, q))
    big.ops[:: 16] = 2
    pkg.test_fail_allocations(1, skip)
    try:
        with pytest.raises(pkg.PiError) as ei:
            run_batch(idx, big)
    finally:
        pkg.test_fail_allocations(0)
    assert ei.value.code == pkg.PI_ERR_OOM
    assert_state_equal(idx, orc, "after the refused batch")
    for i, b in enumerate([inserts(99, 600_000, 40_000), big, inserts(99, 700_000, 200_000)]):
        assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals), f"batch {i}")
    assert_state_equal(idx, orc, "end")
    idx.close()
    orc.close()
