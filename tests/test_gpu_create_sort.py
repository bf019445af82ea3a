"""The bulk build's sort: four passes on the leading varying bytes, then the pairs whose keys agree
on them -- short runs with the passes, a few long ones one by one, many of them by sorting every
byte. The exported pairs are compared with a stable sort of the input in which the last
occurrence of a key wins."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import make_index

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    from paper_1601_00159_gb300 import build, load_library
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return load_library()


def _keys(kind, n, s):
    low = wl.u64_stream(s, 0, n) & np.uint64((1 << 24) - 1)
    lead = wl.bounded(s, n, n, 16).astype(np.uint64)
    if kind == "pairs":  # leading bytes of about n / 2 values: runs of a few keys
        return (wl.bounded(s, n, n, max(n // 2, 1)).astype(np.uint64) << np.uint64(24)) * np.uint64(0x10001) + low
    if kind == "shared":  # 16 leading values: a few runs of n / 16
        return ((lead & np.uint64(1)) << np.uint64(48)) | ((lead >> np.uint64(1) & np.uint64(1)) << np.uint64(40)) | \
            ((lead >> np.uint64(2) & np.uint64(1)) << np.uint64(32)) | ((lead >> np.uint64(3)) << np.uint64(24)) | low
    if kind == "repeated":  # one key in half of the pairs, another of its prefix once
        k = wl.u64_stream(s, 0, n) >> np.uint64(1)
        k = np.where(lead < 8, np.uint64(0x1234567812345678), k)
        k[n // 2] = np.uint64(0x1234567812345679)
        return k
    return wl.u64_stream(s, 0, n) >> np.uint64(1)


@pytest.mark.parametrize("kind", ["wide", "pairs", "shared", "repeated"])
@pytest.mark.parametrize("n", [33, 4097, 40000, 300000, (1 << 20) + 77])
def test_create_orders_pairs(kind, n):
    s = wl.stream_seed(n, 90)
    keys = _keys(kind, n, s).astype(np.uint64)
    vals = wl.u64_stream(s, 3 * n, n)
    idx = make_index(keys, vals, 0.25, 4)
    k, v = idx.export()
    order = np.argsort(keys, kind="stable")
    sk = keys[order]
    last = np.append(sk[1:] != sk[:-1], True)
    assert np.array_equal(k.cpu().numpy().view(np.uint64), sk[last])
    assert np.array_equal(v.cpu().numpy().view(np.uint64), vals[order][last])
    assert idx.size() == int(last.sum()) and idx.status() == 0
    assert idx.export()[0].numel() == int(last.sum())
    idx.close()
