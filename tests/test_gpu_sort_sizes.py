"""The batch sort where its paths change: radix passes with a look-back up to 2^20 queries (tiles
of 2048 and, from 2^19, of 4096), counted passes above; digit counts from the packing when the
passes start at key byte 4, from the plan kernel otherwise. Against the oracle."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_results_equal, make_index, run_batch

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


@pytest.mark.parametrize("passes", [0, 3, 8])
@pytest.mark.parametrize("kind", ["wide", "dense", "hot"])
def test_sizes(orc_mod, kind, passes):
    n = 20000
    number = np.arange(n, dtype=np.uint64)
    keys = number * np.uint64(3) if kind == "dense" else wl.distinct_keys(70, number)
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 5, {"sort_passes": passes})
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 5)
    for c, q in enumerate([(1 << 15) + 1, (1 << 19) - 1, (1 << 19) + 4097, 1 << 20, (1 << 20) + 1]):
        s = wl.stream_seed(c, 71)
        i = wl.bounded(s, 0, q, n)
        if kind == "hot":  # half the batch on one key, a quarter on a few
            u = wl.bounded(s, q, q, 4)
            i = np.where(u < 2, 7, np.where(u == 2, i % 5, i))
        k = keys[i] + (wl.bounded(s, 2 * q, q, 8) == 0).astype(np.uint64)  # some misses
        ops = np.where(wl.bounded(s, 3 * q, q, 10) < 8, 0, 1 + wl.bounded(s, 4 * q, q, 2)).astype(np.uint8)
        odd = wl.bounded(s, 5 * q, q, 100)
        ops = np.where(odd == 0, np.uint8(9), ops).astype(np.uint8)
        k = np.where(odd == 1, wl.RESERVED_KEY, k).astype(np.uint64)
        b = wl.Batch(ops, k, wl.u64_stream(s, 6 * q, q))
        assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals), f"{kind} {q}")
    assert idx.status() == 0
    idx.close()
    orc.close()


@pytest.mark.parametrize("q", [5000, 70001, (1 << 20) + 6])
@pytest.mark.parametrize("shift", [1, 3])
def test_misaligned_arrays(orc_mod, q, shift):
    """Views that start at odd elements: no 16-byte key loads, no word-wide op loads."""
    import torch
    from tests.parity import results_np, to_dev
    n = 9000
    keys = wl.distinct_keys(72, np.arange(n))
    idx = make_index(keys, keys, 0.5, 5)
    orc = orc_mod.Oracle(keys, keys, 0.5, 5)
    s = wl.stream_seed(q, 73)
    ops = wl.bounded(s, 0, q, 4).astype(np.uint8)
    k = keys[wl.bounded(s, q, q, n)]
    b = wl.Batch(ops, k, wl.u64_stream(s, 2 * q, q))
    pad = lambda a, dt: to_dev(np.concatenate([np.zeros(shift, a.dtype), a]), dt)[shift:]  # noqa: E731
    got = idx.execute(pad(b.ops, torch.uint8), pad(b.keys, torch.int64), pad(b.vals, torch.int64))
    assert_results_equal(results_np(got), orc.execute(b.ops, b.keys, b.vals), f"q {q}")
    idx.close()
    orc.close()
