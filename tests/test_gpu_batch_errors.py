"""An index in error: a batch that the device refuses still ends by bringing the device's state to the
host, whichever of the merge's blocks see the error, so the next call reports it."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_state_equal, make_index, run_batch

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


@pytest.mark.parametrize("bits,code", [(1, -4), (2, -3)])
@pytest.mark.parametrize("op", [0, 1, 2])
@pytest.mark.parametrize("q", [500, 40000])
@pytest.mark.parametrize("before", [0, 70])  # 70: more batches than the mailbox ring has slots
def test_index_in_error_is_reported(orc_mod, bits, code, op, q, before):
    import torch
    import paper_1601_00159_gb300 as pkg
    n = 50_000
    keys = wl.distinct_keys(101, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 15)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 15)
    k = wl.distinct_keys(101, np.uint64(100_000) + np.arange(q, dtype=np.uint64)) if op == 1 else keys[:q]
    b = wl.Batch(np.full(q, op, np.uint8), k, k)
    none = wl.Batch(np.zeros(300, np.uint8), keys[:300], keys[:300])
    for _ in range(before):
        run_batch(idx, none)
    torch.cuda.synchronize()
    pkg.test_set_error(idx, bits)
    run_batch(idx, b)  # the host does not know yet
    for _ in range(3):
        with pytest.raises(pkg.PiError) as ei:
            run_batch(idx, none)
        assert ei.value.code == code
    assert idx.status() == code
    pkg.test_set_error(idx, 0)
    assert_state_equal(idx, orc)  # nothing of the refused batch was applied
    idx.close()
    orc.close()
