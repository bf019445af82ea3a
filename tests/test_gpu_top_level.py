"""H, the number of levels (Definition 1), when the levels that come and go lie below the lowest built
one, so that no batch lays the index layer out anew, and with the deferred rebuild policy."""
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


@pytest.mark.parametrize("cfg", [{"lowest_level": 16}, {"lowest_level": 4}, {"lowest_level": 4, "rebuild_policy": 1}])
@pytest.mark.parametrize("multi", [False, True])
def test_top_level_follows_the_live_keys(orc_mod, cfg, multi):
    import torch
    from paper_1601_00159_gb300 import MultiSet
    from tests.parity import results_np, to_dev
    keys = wl.distinct_keys(140, np.arange(300))
    idx = make_index(keys, keys, 0.5, 6, cfg)
    orc = orc_mod.Oracle(keys, keys, 0.5, 6)
    ms = MultiSet([idx]) if multi else None
    seen = set()
    by_level = [orc.level(l) for l in range(2, orc.num_levels() + 1)]
    steps = [(2, by_level[i]) for i in range(len(by_level) - 1, -1, -1)] + [(1, lv) for lv in by_level[::-1]]
    for op, k in steps:
        b = wl.Batch(np.full(len(k), op, np.uint8), k, k)
        if multi:
            dev = [to_dev(b.ops, torch.uint8), to_dev(b.keys, torch.int64), to_dev(b.vals, torch.int64),
                   torch.empty((len(k), 2), dtype=torch.int64, device="cuda")]
            ms.execute([(0, *dev)])
            got = results_np(dev[3])
        else:
            got = run_batch(idx, b)
        assert_results_equal(got, orc.execute(b.ops, b.keys, b.vals))
        top = max(orc.num_levels(), 1)
        assert idx.num_levels() == top and idx.info()["top_level"] == top
        assert idx.info()["level_size"][1] == idx.size() == len(orc.export()[0])
        seen.add(top)
    assert len(seen) > 3 and 1 in seen
    if multi:
        ms.close()
    idx.close()
    orc.close()
