"""The rebuild of a small batch, whose scans and change lists are made inside the writing kernel:
storage sizes around a scan chunk (1024 tiles of 4096 nodes), a batch of new keys (every level
from the storage layer) and one of deletes and revivals (every level from the one before). The
levels equal those of an index built from the same keys, and a batch above the limit, which has
a kernel of its own for the scans, leaves the same."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import PI_OP_DELETE, PI_OP_INSERT
from paper_1601_00159_gb300 import workloads as wl
from tests.parity import make_index

pytestmark = pytest.mark.gpu

CHUNK = 1024 * 4096
SMALL = 1 << 15


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    from paper_1601_00159_gb300 import build, load_library
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return load_library()


def _run(idx, op, keys):
    import torch
    k = torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda()
    idx.execute(torch.full((len(keys),), op, dtype=torch.uint8, device="cuda"), k, k)


def _levels(idx):
    info = idx.info()
    return [tuple(t.cpu().numpy() for t in idx.export_level(l))
            for l in range(info["bottom_built"], info["top_level"] + 1)]


def _check(idx, p, seed):
    """Level keys as a bulk build of the live keys has them; each down entry is its key's place."""
    keys, vals = idx.export()
    ref = make_index(keys.cpu().numpy().view(np.uint64), vals.cpu().numpy().view(np.uint64), p, seed)
    got, want = _levels(idx), _levels(ref)
    assert idx.status() == 0 and len(got) == len(want)
    below = idx.export_storage()[0].cpu().numpy()
    for g, w in zip(got, want):
        assert np.array_equal(g[0], w[0])
        assert np.array_equal(below[g[1].view(np.uint32).astype(np.int64)], g[0])
        below = g[0]
    ref.close()


@pytest.mark.parametrize("q", [1, 1000, SMALL, SMALL + 1])
@pytest.mark.parametrize("n", [3000, CHUNK - 1000, CHUNK + 3])
def test_levels_after_small_batches(n, q):
    q = min(q, n // 2)
    keys = wl.distinct_keys(11, np.arange(n + q, dtype=np.uint64))
    idx = make_index(keys[:n], keys[:n], 0.25, 5)
    _run(idx, PI_OP_INSERT, keys[n:])
    _check(idx, 0.25, 5)
    _run(idx, PI_OP_DELETE, keys[:q])
    _check(idx, 0.25, 5)
    _run(idx, PI_OP_INSERT, keys[:q:2])
    _check(idx, 0.25, 5)
    idx.close()
