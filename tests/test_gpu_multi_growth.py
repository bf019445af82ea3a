"""Growth of an index's arrays under the batching form."""
import time

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


def dev_batch(b):
    import torch
    return (to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
            torch.empty((len(b), 2), dtype=torch.int64, device="cuda"))


def test_index_layer_grows_once(orc_mod):
    """An index layer that outgrew its capacity is grown by one call; the calls after it do not
    synchronise to look again, though none of them lays the levels out anew."""
    import torch
    from paper_1601_00159_gb300 import MultiSet
    keys = wl.distinct_keys(95, np.arange(20000))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 5, {"index_capacity": 64})
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 5)
    ms = MultiSet([idx])
    small = idx.info()["index_capacity"]
    b = wl.Batch(np.zeros(700, np.uint8), keys[:700], keys[:700])
    dev = dev_batch(b)
    for _ in range(4):
        ms.execute([(0, *dev)])
        torch.cuda.synchronize()
    assert idx.info()["index_capacity"] > small
    for _ in range(2):  # (the look at the sizes above is not part of what is timed)
        ms.execute([(0, *dev)])
        torch.cuda.synchronize()
    t0 = time.perf_counter()
    torch.cuda._sleep(400_000_000)  # some 200 ms on the stream
    ms.execute([(0, *dev)])
    t1 = time.perf_counter()
    torch.cuda.synchronize()
    t2 = time.perf_counter()
    assert t1 - t0 < 0.5 * (t2 - t0), f"the call waited: {t1 - t0:.3f} of {t2 - t0:.3f} s"
    assert_results_equal(results_np(dev[3]), orc.execute(b.ops, b.keys, b.vals))
    ms.close()
    assert_state_equal(idx, orc)
    idx.close()
    orc.close()


def mixed(keys, seed, q, inserts):
    s = wl.stream_seed(seed, 96)
    k = np.concatenate([keys[wl.bounded(s, 0, q - inserts, len(keys))], wl.u64_stream(s, q, inserts) >> np.uint64(1)])
    return wl.Batch(np.repeat(np.array([0, 1], np.uint8), [q - inserts, inserts]), k, wl.u64_stream(s, 2 * q, q))


@pytest.mark.parametrize("fails", [1, 2])
@pytest.mark.parametrize("skip", [0, 1, 2])
@pytest.mark.parametrize("needed", [False, True])
def test_growth_that_fails_part_way(orc_mod, needed, skip, fails):
    """An index that comes near its capacity gets more room than the call needs. Whichever of that
    growth's allocations fails, the call does without the room when it does not need it, and
    takes just what it needs when it does; only a failure of that refuses it. The set and the plain
    path are right afterwards."""
    import torch
    import paper_1601_00159_gb300 as pkg
    n, q = 70_000, 50_000
    keys = wl.distinct_keys(96, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 13)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 13)
    ms = pkg.MultiSet([idx])
    cap = idx.info()["storage_capacity"]

    def check(b, dev, what):
        torch.cuda.synchronize()
        assert_results_equal(results_np(dev[3]), orc.execute(b.ops, b.keys, b.vals), what)

    calls = [mixed(keys, 1, q, 0), mixed(keys, 2, 20_000, 20_000 if needed else 0),
             mixed(keys, 3, q, q if needed else 1000)]
    devs = [dev_batch(b) for b in calls]
    ms.execute([(0, *devs[0])])  # the class's scratch
    check(calls[0], devs[0], "call 0")
    torch.cuda._sleep(100_000_000)  # call 1 stays in flight: its queries count as possible nodes
    ms.execute([(0, *devs[1])])
    assert (n + len(calls[1]) + q > cap) and (needed == (n + int(calls[1].ops.sum()) + q > cap))
    pkg.test_fail_allocations(fails, skip)
    try:
        refused = False
        try:
            ms.execute([(0, *devs[2])])
        except pkg.PiError as e:
            assert e.code == pkg.PI_ERR_OOM
            refused = True
    finally:
        pkg.test_fail_allocations(0)
    # the first failure is the room's; a second one meets what the batch needs, if it needs any
    assert refused == (needed and fails == 2)
    check(calls[1], devs[1], "call 1")
    if refused:
        assert idx.info()["storage_capacity"] == cap
        ms.execute([(0, *devs[2])])
    check(calls[2], devs[2], "call 2")
    assert (idx.info()["storage_capacity"] > cap) == needed
    for i in range(2):
        b = mixed(keys, 20 + i, 60_000, 40_000)
        dev = dev_batch(b)
        idx.execute(*dev)
        check(b, dev, f"plain {i}")
        b = mixed(keys, 30 + i, q, 30_000)
        dev = dev_batch(b)
        ms.execute([(0, *dev)])
        check(b, dev, f"set {i}")
    ms.close()
    assert_state_equal(idx, orc)
    idx.close()
    orc.close()


@pytest.mark.parametrize("alone", [True, False])
def test_call_refused_after_an_index_grew(orc_mod, alone):
    """A call in which one index grows and the next cannot is refused. The set's later calls, on the
    first index alone or on both, work on its new arrays."""
    import torch
    import paper_1601_00159_gb300 as pkg
    n, q = 70_000, 100_000
    keys = [wl.distinct_keys(102 + i, np.arange(n)) for i in range(2)]
    idx = [make_index(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]
    orc = [orc_mod.Oracle(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]
    ms = pkg.MultiSet(idx)
    caps = [x.info()["storage_capacity"] for x in idx]
    assert n + q > max(caps)

    def call(bs):
        devs = [dev_batch(b) for b in bs]
        ms.execute([(i, *d) for i, d in enumerate(devs)])
        torch.cuda.synchronize()
        for i, (b, d) in enumerate(zip(bs, devs)):
            assert_results_equal(results_np(d[3]), orc[i].execute(b.ops, b.keys, b.vals), f"index {i}")

    call([mixed(k, 1, n // 2, 0) for k in keys])
    bs = [mixed(k, 2 + i, q, q) for i, k in enumerate(keys)]
    pkg.test_fail_allocations(2, 3)  # the first index's storage, look-back words and counts succeed
    try:
        with pytest.raises(pkg.PiError) as ei:
            ms.execute([(i, *dev_batch(b)) for i, b in enumerate(bs)])
    finally:
        pkg.test_fail_allocations(0)
    assert ei.value.code == pkg.PI_ERR_OOM
    grown = [x.info()["storage_capacity"] for x in idx]
    assert grown[0] > caps[0] and grown[1] == caps[1]
    call(bs[:1] if alone else bs)
    call([mixed(k, 7 + i, q, q // 2) for i, k in enumerate(keys)])
    ms.close()
    for x, o in zip(idx, orc):
        assert_state_equal(x, o)
        x.close()
        o.close()
