"""Small batches: tiles sorted in shared memory and placed by rank, against the radix path.

A batch of at most 2^15 queries is sorted tile by tile (1024 queries) and looked up query by
query; PI_TEST_SORT_PREFIX(4) keeps the same batch on the radix passes and the
level-synchronous descent. Both must equal the oracle at the tile edges, with more tiles than
a look-up block has warps, with hot keys whose runs cross tiles, with invalid queries, and on
an index without any built level.
"""
import numpy as np
import pytest

from paper_1601_00159_gb300 import PI_TEST_SORT_PREFIX
from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_results_equal, assert_state_equal, make_index, run_batch

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


@pytest.mark.parametrize("flags", [0, PI_TEST_SORT_PREFIX(4)])
@pytest.mark.parametrize("key_range", [3, 900, 1 << 62])
@pytest.mark.parametrize("n", [0, 20, 30000])
def test_tile_edges(orc_mod, n, key_range, flags):
    sizes = [1, 7, 9, 33, 63, 65, 1023, 1024, 1025, 2048, 8191, 8193, (1 << 15) - 1, 1 << 15, (1 << 15) + 1]
    s = wl.stream_seed(n + key_range % 1000003, 17)
    keys = wl.bounded(s, 0, n, min(key_range, 1 << 31)).astype(np.uint64) if key_range < (1 << 31) else \
        wl.u64_stream(s, 0, n) >> np.uint64(2)
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 9, {"test_flags": flags} if flags else None)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 9)
    for c, q in enumerate(sizes):
        sb = wl.stream_seed(c, 18)
        ops = wl.bounded(sb, 0, q, 3).astype(np.uint8)
        if key_range < (1 << 31):
            bk = wl.bounded(sb, q, q, key_range).astype(np.uint64)
        else:
            bk = wl.u64_stream(sb, q, q) >> np.uint64(2)
            if n:
                bk = np.where(wl.bounded(sb, 2 * q, q, 2) == 0, keys[wl.bounded(sb, 3 * q, q, n)], bk)
        odd = wl.bounded(sb, 4 * q, q, 50)
        ops = np.where(odd == 0, np.uint8(3), ops).astype(np.uint8)
        bk = np.where(odd == 1, wl.RESERVED_KEY, bk)
        bk = np.where(odd == 2, wl.RESERVED_KEY - np.uint64(1), bk)
        b = wl.Batch(ops, bk.astype(np.uint64), wl.u64_stream(sb, 5 * q, q))
        assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals), f"n {n} q {q}")
    assert_state_equal(idx, orc, f"n {n} range {key_range}")
    idx.close()
    orc.close()
