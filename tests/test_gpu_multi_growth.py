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
