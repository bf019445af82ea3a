"""Calls of one set on different streams, on indices that they do not share: the set's queue and
scratch are one, so they run one after another. Every result and the final pairs equal the oracle's."""
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


@pytest.mark.parametrize("classes", [[(32, 8, 8)], [(32, 16, 8, 2)]])
def test_disjoint_calls_on_two_streams(orc_mod, classes):
    import torch
    from paper_1601_00159_gb300 import MultiSet
    n, q, members = 20_000, 20_000, ([0, 1], [2, 3, 4])
    keys = [wl.distinct_keys(110 + i, np.arange(n)) for i in range(5)]
    idx = [make_index(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]
    orc = [orc_mod.Oracle(k, wl.splitmix64(k), 0.25, i) for i, k in enumerate(keys)]
    ms = MultiSet(idx, classes)
    runs = []
    for step in range(12):
        run = []
        for i in members[step % 2]:
            s = wl.stream_seed(110, 10 * step + i)
            k = np.concatenate([keys[i][wl.bounded(s, 0, q // 2, n)], wl.u64_stream(s, q, q // 2) >> np.uint64(1)])
            b = wl.Batch(np.tile(np.array([0, 1, 2, 1], np.uint8), q // 4), k, wl.u64_stream(s, 2 * q, q))
            run.append((i, b, (to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
                               torch.empty((q, 2), dtype=torch.int64, device="cuda"))))
        runs.append(run)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for step, run in enumerate(runs):
        ms.execute([(i, *dev) for i, _, dev in run], stream=streams[step % 2])
    torch.cuda.synchronize()
    for step, run in enumerate(runs):
        for i, b, dev in run:
            assert_results_equal(results_np(dev[3]), orc[i].execute(b.ops, b.keys, b.vals), f"step {step} index {i}")
    ms.close()
    for x, o in zip(idx, orc):
        assert_state_equal(x, o)
        x.close()
        o.close()
