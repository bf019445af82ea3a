"""The 32-bit epoch that tags look-back descriptors starts again from one after some 10^9 batches, with
the descriptors cleared: not under the background rebuild of the batch before, which may still be
looking back over them."""
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


@pytest.mark.parametrize("n,q", [(20_000, 500), (200_000, 40_000), (1_000_000, 600_000)])
def test_batches_across_the_wrap(orc_mod, n, q):
    import torch
    import paper_1601_00159_gb300 as pkg
    keys = wl.distinct_keys(150, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 8, {"storage_capacity": 4_000_000})
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 8)
    runs = []
    for step in range(8):
        s = wl.stream_seed(150, step)
        k = np.concatenate([keys[wl.bounded(s, 0, q - q // 8, n)], wl.u64_stream(s, q, q // 8) >> np.uint64(1)])
        b = wl.Batch(wl.bounded(s, 2 * q, q, 3).astype(np.uint8), k, wl.u64_stream(s, 3 * q, q))
        runs.append((b, [to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
                         torch.empty((q, 2), dtype=torch.int64, device="cuda")]))
    torch.cuda.synchronize()
    for step, (b, dev) in enumerate(runs):  # back to back: a rebuild is in flight when the next batch starts
        if step % 2 == 1:
            pkg.test_set_epoch(idx, 2 ** 32 - 40)
        idx.execute(*dev)
    torch.cuda.synchronize()
    assert idx.status() == 0
    for step, (b, dev) in enumerate(runs):
        assert_results_equal(results_np(dev[3]), orc.execute(b.ops, b.keys, b.vals), f"batch {step}")
    assert_state_equal(idx, orc)
    idx.close()
    orc.close()
