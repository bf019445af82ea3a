"""Range queries as runs of nodes: a warp takes 1 to 32 consecutive queries, by their number.

Empty, single-key, long and overlapping ranges side by side, with and without delete-flagged
nodes, at query counts on either side of the points where a warp takes more of them; and a
capacity that cuts a run in the middle.
"""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import make_index, run_batch, to_dev

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


@pytest.mark.parametrize("n", [0, 40, 60000])
@pytest.mark.parametrize("deleted", [False, True])
@pytest.mark.parametrize("q", [1, 17, 255, 4800, 9800, 40000, 160000])
def test_runs(orc_mod, n, deleted, q):
    import torch
    keys = np.sort(wl.distinct_keys(60, np.arange(n)))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 3)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 3)
    if deleted and n:
        dk = keys[wl.bounded(wl.stream_seed(61, 0), 0, n // 8, n)]
        b = wl.Batch(np.full(len(dk), 2, np.uint8), dk, np.zeros(len(dk), np.uint64))
        run_batch(idx, b)
        orc.execute(b.ops, b.keys, b.vals)
    s = wl.stream_seed(q, 62)
    lo = wl.u64_stream(s, 0, q) >> np.uint64(1)
    step = np.uint64((1 << 63) // max(n, 1))
    span = wl.bounded(s, q, q, 12).astype(np.uint64) * step
    long = np.uint64(min(700 * int(step), (1 << 63) - 1))
    span = np.where(wl.bounded(s, 2 * q, q, 200) == 0, long, span)  # a few long ones
    if n:
        at = keys[wl.bounded(s, 3 * q, q, n)]
        lo = np.where(wl.bounded(s, 4 * q, q, 3) == 0, at, lo)  # bounds that are keys
    hi = lo + span
    empty = wl.bounded(s, 5 * q, q, 5) == 0
    hi = np.where(empty, lo - np.uint64(1), hi)
    lo[0], hi[0] = 0, wl.RESERVED_KEY
    eo, ek, ev = orc.range(lo.astype(np.uint64), hi.astype(np.uint64))
    total = int(eo[-1])
    offs, k, v = idx.range_search(to_dev(lo, torch.int64), to_dev(hi, torch.int64), cap=max(total, 1))
    assert np.array_equal(offs.cpu().numpy().view(np.uint64), eo)
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ek)
    assert np.array_equal(v.cpu().numpy().view(np.uint64), ev)
    if total > 3:  # a capacity inside the output: whole queries below it are written, nothing past it
        cap = 2 * total // 3
        dlo, dhi = to_dev(lo, torch.int64), to_dev(hi, torch.int64)
        out = torch.full((2, cap + 1), -7, dtype=torch.int64, device="cuda")
        assert idx.lib.pi_range_search(idx._h, dlo.data_ptr(), dhi.data_ptr(), q, offs.data_ptr(), out[0].data_ptr(),
                                       out[1].data_ptr(), cap, None) == 0
        torch.cuda.synchronize()
        fit = int(eo[np.searchsorted(eo, cap, side="right") - 1])
        got = out.cpu().numpy().view(np.uint64)
        assert np.array_equal(offs.cpu().numpy().view(np.uint64), eo)
        assert np.array_equal(got[0, :fit], ek[:fit]) and np.array_equal(got[1, :fit], ev[:fit])
        assert (out[:, fit:] == -7).all()
    assert idx.status() == 0
    idx.close()
    orc.close()
