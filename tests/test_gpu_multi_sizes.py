"""The host's view of index sizes between batching-form calls: calls of two sets that share an index,
and plain batches between them, without a synchronisation, every batch all new keys, past the
initial capacity. Every result and the final pairs equal the oracle's."""
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


@pytest.mark.parametrize("q", [900, 30000])
def test_two_sets_and_plain_batches(orc_mod, q):
    import torch
    from paper_1601_00159_gb300 import MultiSet
    idx, orc = [], []
    for i in range(3):
        keys = wl.distinct_keys(80 + i, np.arange(2000))
        idx.append(make_index(keys, wl.splitmix64(keys), 0.25, i))
        orc.append(orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, i))
    sets = [(MultiSet([idx[0], idx[1]], [(32, 16, 8, 2)]), [0, 1]), (MultiSet([idx[1], idx[2]]), [1, 2])]
    runs = []
    for step in range(8):
        def batch(i):
            s = wl.stream_seed(step * 10 + i, 81)
            n = q if (step + i) % 3 else q // 7
            k = wl.distinct_keys(80 + i, np.uint64(10_000 + step * 100_000) + np.arange(n, dtype=np.uint64))
            return wl.Batch(np.full(n, 1, np.uint8), k, wl.u64_stream(s, 0, n))
        todo = []
        if step % 3 == 2:
            todo = [(1, batch(1), None)]
        else:
            ms, members = sets[step % 2]
            todo = [(i, batch(i), j) for j, i in enumerate(members)]
        desc = []
        for i, b, j in todo:
            dev = (to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
                   torch.empty((len(b), 2), dtype=torch.int64, device="cuda"))
            runs.append((step, i, b, dev))
            if j is None:
                idx[i].execute(*dev)
            else:
                desc.append((j, *dev))
        if desc:
            ms.execute(desc)
    torch.cuda.synchronize()
    for step, i, b, dev in runs:
        assert_results_equal(results_np(dev[3]), orc[i].execute(b.ops, b.keys, b.vals), f"step {step} index {i}")
    for i in range(3):
        assert_state_equal(idx[i], orc[i], f"index {i}")
    for ms, _ in sets:
        ms.close()
    for x in idx + orc:
        x.close()
