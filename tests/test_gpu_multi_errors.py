"""A set with an index in error: the batching form reports the index's sticky error on one of the
next calls, as the single-index path does, and never returns PI_OK for work that the device refused
once the call that met the error has finished."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_results_equal, assert_state_equal, make_index, results_np, to_dev

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


def make_set(n=3000, count=3):
    keys = [wl.distinct_keys(90 + i, np.arange(n)) for i in range(count)]
    return keys, [make_index(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]


def search_and_insert(keys, seed, q=500):
    s = wl.stream_seed(seed, 91)
    k = np.concatenate([keys[wl.bounded(s, 0, q, len(keys))], wl.u64_stream(s, q, q) >> np.uint64(1)])
    return wl.Batch(np.repeat(np.array([0, 1], np.uint8), q), k, wl.u64_stream(s, 2 * q, 2 * q))


def dev_batch(b):
    import torch
    return (to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
            torch.empty((len(b), 2), dtype=torch.int64, device="cuda"))


@pytest.mark.parametrize("classes", [[(32, 8, 8)], [(32, 16, 8, 2)]])
@pytest.mark.parametrize("calls_before", [0, 1, 3])
def test_index_in_error_is_reported(orc_mod, classes, calls_before):
    import torch
    import paper_1601_00159_gb300 as pkg
    keys, idx = make_set()
    orc = [orc_mod.Oracle(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]
    ms = pkg.MultiSet(idx, classes)

    def call(step):
        bs = [search_and_insert(k, 10 * step + i) for i, k in enumerate(keys)]
        devs = [dev_batch(b) for b in bs]
        ms.execute([(i, *d) for i, d in enumerate(devs)])
        torch.cuda.synchronize()
        return bs, devs

    for step in range(calls_before):
        for i, (b, d) in enumerate(zip(*call(step))):
            assert_results_equal(results_np(d[3]), orc[i].execute(b.ops, b.keys, b.vals), f"step {step} index {i}")
    pkg.test_set_error(idx[1], 1)
    try:  # the host may not know of the error yet; the device refuses that index's batch
        bs, devs = call(50)
        for i in (0, 2):
            b = bs[i]
            assert_results_equal(results_np(devs[i][3]), orc[i].execute(b.ops, b.keys, b.vals), f"index {i}")
    except pkg.PiError as e:
        assert e.code == pkg.PI_ERR_TIMEOUT
    for step in (51, 52, 53):  # the call has finished: every later one reports it
        with pytest.raises(pkg.PiError) as ei:
            call(step)
        assert ei.value.code == pkg.PI_ERR_TIMEOUT
    with pytest.raises(pkg.PiError) as ei:
        idx[1].execute(*dev_batch(search_and_insert(keys[1], 60)))
    assert ei.value.code == pkg.PI_ERR_TIMEOUT
    ms.close()
    pkg.test_set_error(idx[1], 0)
    assert [x.status() for x in idx] == [0, 0, 0]
    for x, o in zip(idx, orc):  # the other indices ran, the refused one is as it was
        assert_state_equal(x, o)
        x.close()
        o.close()
