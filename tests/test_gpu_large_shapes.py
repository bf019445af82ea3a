"""Branches that only large or lopsided shapes take: a run of equal keys longer than the nearest blocks'
marks reach, tiles whose stretch of the lowest built level does not fit a window, windows over the
storage layer itself, merges of so many nodes that a CTA finds its cuts in groups, range slices
copied one at a time, and slices long enough to be counted by a whole warp. Everything is compared with the oracle, or, at 2^28 keys, with the
same update done by sorting."""
import numpy as np
import pytest

from paper_1601_00159_gb300 import workloads as wl
from tests.parity import assert_results_equal, assert_state_equal, make_index, run_batch, to_dev

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


def check(orc_mod, keys, p, batches, cfg=None, **state):
    idx = make_index(keys, wl.splitmix64(keys), p, 21, cfg)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), p, 21)
    for i, b in enumerate(batches):
        assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals), f"batch {i}")
    assert_state_equal(idx, orc, **state)
    idx.close()
    orc.close()


@pytest.mark.parametrize("q,hot", [((1 << 20) + 77, 300_000), (1 << 20, 33_000), (1 << 18, 100_000)])
@pytest.mark.parametrize("write", ["none", "first", "last"])
@pytest.mark.parametrize("flags", [0, 1])  # 1: without windows
def test_long_run_of_searches(orc_mod, q, hot, write, flags):
    keys = wl.distinct_keys(120, np.arange(60_000))
    s = wl.stream_seed(q, 121)
    k = keys[wl.bounded(s, 0, q, len(keys))]
    hk = keys[777]
    at = np.sort(np.argsort(wl.u64_stream(s, q, q))[:hot])  # where the hot key's queries arrive
    k[at] = hk
    ops = np.where(wl.bounded(s, 2 * q, q, 50) == 0, 1, 0).astype(np.uint8)  # other keys are written too
    ops[k == hk] = 0
    at = np.nonzero(k == hk)[0]
    if write != "none":
        ops[at[0] if write == "first" else at[-1]] = 1
    b = wl.Batch(ops, k, wl.u64_stream(s, 3 * q, q))
    gone = wl.Batch(np.where(k == hk, 2, 0).astype(np.uint8), k, b.vals)  # one delete, then searches
    gone.ops[at[1:]] = 0
    check(orc_mod, keys, 0.25, [b, gone, b], {"test_flags": flags} if flags else None)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("write", [None, 1000, 5_000_000])
def test_batch_of_one_key(write, flags):
    """A run over more groups of marks than one step of the look-back takes."""
    import torch
    n, q = 1 << 20, (1 << 24) + 33
    keys = wl.distinct_keys(128, np.arange(n))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 23, {"test_flags": flags} if flags else None)
    old = int(wl.splitmix64(keys[7:8]).view(np.int64)[0])
    ops = torch.zeros(q, dtype=torch.uint8, device="cuda")
    k = to_dev(keys[7:8], torch.int64).expand(q).contiguous()
    vals = torch.full((q,), 4711, dtype=torch.int64, device="cuda")
    want = torch.full((q,), old, dtype=torch.int64, device="cuda")
    if write is not None:
        ops[write] = 1
        want[write + 1:] = 4711
    r = idx.execute(ops, k, vals)
    assert torch.equal(r[:, 0], want) and bool((r[:, 1] == 1).all())
    if write is not None:  # then a delete, after which the key is absent
        ops[write] = 2
        r = idx.execute(ops, k, vals)
        assert bool((r[: write + 1, 0] == 4711).all()) and bool((r[: write + 1, 1] == 1).all())
        assert not bool(r[write + 1:].any())
    assert idx.status() == 0
    idx.close()


@pytest.mark.parametrize("q", [1 << 19, (1 << 20) + 5])
def test_stretch_longer_than_a_window(orc_mod, q):
    """Most queries fall on a narrow range of keys, the others spread thinly over a large index."""
    n = 1 << 23
    keys = np.sort(wl.distinct_keys(122, np.arange(n)))
    s = wl.stream_seed(q, 123)
    narrow = keys[n // 3 + wl.bounded(s, 0, q, 5000).astype(np.int64)]
    wide = np.where(wl.bounded(s, q, q, 2) == 0, keys[wl.bounded(s, 2 * q, q, n)], wl.u64_stream(s, 3 * q, q) >> np.uint64(1))
    k = np.where(wl.bounded(s, 4 * q, q, 64) == 0, wide, narrow)
    b = wl.Batch(wl.bounded(s, 5 * q, q, 3).astype(np.uint8), k, wl.u64_stream(s, 6 * q, q))
    check(orc_mod, keys, 0.25, [b], {"lowest_level": 3}, check_levels=False)


@pytest.mark.parametrize("n", [0, 1, 5000, 300_000])
def test_windows_without_a_built_level(orc_mod, n):
    q = 1 << 19
    keys = wl.distinct_keys(124, np.arange(n))
    s = wl.stream_seed(n, 125)
    miss = wl.u64_stream(s, 0, q) >> np.uint64(1)
    k = np.where(wl.bounded(s, q, q, 2) == 0, keys[wl.bounded(s, 2 * q, q, n)], miss) if n else miss
    ops = np.where(wl.bounded(s, 3 * q, q, 4) == 0, 1 + wl.bounded(s, 4 * q, q, 2), 0).astype(np.uint8)
    search = wl.Batch(np.zeros(q, np.uint8), k, k)
    few = wl.Batch(np.where(np.arange(q) % 64 == 0, ops, 0).astype(np.uint8), k, wl.u64_stream(s, 5 * q, q))
    check(orc_mod, keys, 1 / 16, [search, few, search], {"lowest_level": 16})


@pytest.mark.parametrize("flagged", [False, True])
def test_merge_with_cuts_in_groups(flagged):
    """2^28 nodes, some 350 chunks for each CTA of the merge."""
    import torch
    from paper_1601_00159_gb300 import Index
    n, q = 1 << 28, 1 << 20
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    keys = torch.arange(n, dtype=torch.int64, device="cuda") * 16
    idx = Index(keys, keys ^ 12345, 0.25, 22)
    live = torch.ones(n, dtype=torch.bool, device="cuda")
    new = torch.randperm(n // 64, device="cuda", generator=g)[:q] * 1024 + torch.randint(1, 16, (q,), device="cuda", generator=g)
    new[: q // 8] = n * 16 + torch.randperm(q // 8, device="cuda", generator=g) * 3  # past every key
    batch = (torch.ones(q, dtype=torch.uint8, device="cuda"), new, new ^ 999)
    if flagged:
        gone = torch.randperm(n // 4, device="cuda", generator=g)[:q] * 4 + 1
        live[gone] = False
        batch = (torch.cat([batch[0], torch.full((q,), 2, dtype=torch.uint8, device="cuda")]),
                 torch.cat([new, gone * 16]), torch.cat([new ^ 999, gone]))
    order = torch.randperm(batch[0].numel(), device="cuda", generator=g)
    batch = [t[order].contiguous() for t in batch]
    r = idx.execute(*batch)
    assert torch.equal((r[:, 1] & 0xFFFFFFFF) == 1, batch[0] == 2)  # deleted keys were there, new ones were not
    ek = torch.cat([keys[live], new])
    ev = torch.cat([keys[live] ^ 12345, new ^ 999])
    del keys, live
    ek, by = ek.sort()
    ev = ev[by]
    del by
    k, v = idx.export()
    assert torch.equal(k, ek) and torch.equal(v, ev)
    assert idx.status() == 0
    del k, v
    probe = torch.randint(0, n * 16 + 100, (q,), dtype=torch.int64, device="cuda", generator=g)  # through the new levels
    probe[: q // 2] = ek[torch.randint(0, ek.numel(), (q // 2,), device="cuda", generator=g)]
    r = idx.execute(torch.zeros(q, dtype=torch.uint8, device="cuda"), probe, probe)
    at = torch.searchsorted(ek, probe).clamp_(max=ek.numel() - 1)
    hit = ek[at] == probe
    assert torch.equal((r[:, 1] & 0xFFFFFFFF) == 1, hit)
    assert torch.equal(r[:, 0], torch.where(hit, ev[at], torch.zeros_like(probe)))
    idx.close()


@pytest.mark.parametrize("q", [4000, 9800, 40_000, 160_000])
def test_range_slices_one_at_a_time(orc_mod, q):
    import torch
    n = 30_000
    keys = np.sort(wl.distinct_keys(126, np.arange(n)))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 3, {"test_flags": 0x200})
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 3)
    gone = keys[::9]
    b = wl.Batch(np.full(len(gone), 2, np.uint8), gone, gone)
    assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals))
    s = wl.stream_seed(q, 127)
    at = wl.bounded(s, 0, q, n).astype(np.int64)
    span = wl.bounded(s, q, q, 12).astype(np.int64)  # with empty ranges between
    span = np.where(wl.bounded(s, 2 * q, q, 97) == 0, 500, span)
    lo, hi = keys[at], keys[np.minimum(at + span, n - 1)] - np.uint64(1)
    eo, ek, ev = orc.range(lo, hi)
    total = int(eo[-1])
    for cap in (total, 2 * total // 3):
        out = torch.full((2, cap + 1), -7, dtype=torch.int64, device="cuda")
        offs = torch.empty(q + 1, dtype=torch.int64, device="cuda")
        dlo, dhi = to_dev(lo, torch.int64), to_dev(hi, torch.int64)
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


@pytest.mark.parametrize("q", [1, 40, 5000, 160_000])
def test_long_range_slices_with_deleted_nodes(orc_mod, q):
    """Slices of 255 to some thousand 16-byte chunks of state bytes, from any node to any node, among
    short and empty ones."""
    import torch
    n = 60_000
    keys = np.sort(wl.distinct_keys(129, np.arange(n)))
    idx = make_index(keys, wl.splitmix64(keys), 0.25, 3)
    orc = orc_mod.Oracle(keys, wl.splitmix64(keys), 0.25, 3)
    gone = keys[wl.bounded(wl.stream_seed(130, 0), 0, n // 10, n)]
    b = wl.Batch(np.full(len(gone), 2, np.uint8), gone, gone)
    assert_results_equal(run_batch(idx, b), orc.execute(b.ops, b.keys, b.vals))
    s = wl.stream_seed(q, 131)
    at = wl.bounded(s, 0, q, n).astype(np.int64)
    kind = wl.bounded(s, q, q, max(q // 40, 1))  # some forty long ones
    span = np.where(kind == 0, 4000 + wl.bounded(s, 2 * q, q, 50_000).astype(np.int64),
                    wl.bounded(s, 3 * q, q, 30).astype(np.int64))
    edge = kind == 1  # at the limit, from every offset
    span = np.where(edge, 255 * 16 - 20 + wl.bounded(s, 4 * q, q, 40).astype(np.int64), span)
    lo, hi = keys[at], keys[np.minimum(at + span, n - 1)]
    eo, ek, ev = orc.range(lo, hi)
    offs, k, v = idx.range_search(to_dev(lo, torch.int64), to_dev(hi, torch.int64), cap=int(eo[-1]))
    assert np.array_equal(offs.cpu().numpy().view(np.uint64), eo)
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ek)
    assert np.array_equal(v.cpu().numpy().view(np.uint64), ev)
    assert idx.status() == 0
    idx.close()
    orc.close()
