"""Slot tags: one byte per slot that lookups compare first and claims own.

A tag must be 0 exactly where the slot is EMPTY and match the slot's key
elsewhere; a stale byte would hide a key, leak a slot or let two keys claim
one.  The dump's free masks are the zero tags, so the image check compares
tags with words, and finds of every key compare the others.  Sizes sit at the
edges: one to three buckets (both candidates often the same bucket), batches
around the 32 ops of a warp, buckets filled to the last slot, and churn that
reuses every slot many times, in each of the three ways a batch can run.
"""
import numpy as np
import pytest

import oracle
from paper_2510_15095_gb300 import workload as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15095_gb300 import hive
    hive.load_library()
    return hive


def up(H, a):
    return H.to_device_u32(a)


def check(H, t, d, keys):
    v, f = t.find(up(H, keys))
    ev, ef = d.find(keys)
    assert np.array_equal(f.cpu().numpy(), ef) and np.array_equal(H.to_host_u32(v), ev)
    img = t.dump()
    code, where = oracle.check_image(img, img["S"], d, None)
    assert code == 0, f"invariant {code} fails at {where}"


@pytest.mark.parametrize("bs", [16, 32])
@pytest.mark.parametrize("buckets", [1, 2, 3, 5, 64])
@pytest.mark.parametrize("n", [1, 31, 33, 257])
def test_tiny_tables_and_ragged_batches(H, bs, buckets, n):
    t = H.HiveTable(bs * buckets, bucket_slots=bs)
    d = oracle.Dict()
    keys, c = W.take_keys(900 + n, 0, n)
    vals = W.values_for(keys, 1)
    absent, _ = W.take_keys(900 + n, c, n)
    probe = np.concatenate([keys, absent])
    for _ in range(3):
        assert np.array_equal(t.insert(up(H, keys), up(H, vals)).cpu().numpy(),
                              d.insert(keys, vals))
        check(H, t, d, probe)
        er = keys[::2].copy()
        assert np.array_equal(t.erase(up(H, er)).cpu().numpy(), d.erase(er))
        check(H, t, d, probe)
    assert t.check() == 0
    t.close()


@pytest.mark.parametrize("bs", [16, 32])
@pytest.mark.parametrize("way", ["phased", "deferred", "fused"])
def test_churn_keeps_tags_and_words_together(H, bs, way):
    """Batches that erase as many keys as they insert, at 95% load, so that
    every slot changes hands several times and chains run in each batch."""
    big = way == "deferred"  # claims in their own kernel from 2^18 ops on
    slots = 1 << (19 if big else 14)
    rng = np.random.default_rng(bs)
    t = H.HiveTable(slots, bucket_slots=bs)
    d = oracle.Dict()
    live, c = W.take_keys(77, 0, slots * 95 // 100)
    assert np.array_equal(t.insert(up(H, live), up(H, W.values_for(live, 3))).cpu().numpy(),
                          d.insert(live, W.values_for(live, 3)))
    n = slots // 4
    rounds = 4 if big else 12
    for r in range(rounds):
        new, c = W.take_keys(77, c, n)
        ops, keys, vals = W.mixed_batch(rng, live, new, n, n, 2 * n if big else n, seed=r)
        vo, st = t.execute(torch.from_numpy(ops).cuda(), up(H, keys), up(H, vals),
                           fused=way == "fused")
        ev, es = d.execute(ops, keys, vals)
        assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
        live, _ = d.dump()
    check(H, t, d, np.concatenate([live, W.take_keys(77, c, 1000)[0]]))
    assert t.check() == 0
    t.close()


@pytest.mark.parametrize("bs", [16, 32])
def test_every_slot_of_full_buckets(H, bs):
    """Fills a table to the last slot through small inserts (claims, chains,
    stash) and finds every key after each; then empties it."""
    slots = 64 * bs
    t = H.HiveTable(slots, bucket_slots=bs)
    d = oracle.Dict()
    keys, _ = W.take_keys(5, 0, slots)
    vals = W.values_for(keys, 5)
    for part in np.array_split(np.arange(slots), 16):
        assert np.array_equal(t.insert(up(H, keys[part]), up(H, vals[part])).cpu().numpy(),
                              d.insert(keys[part], vals[part]))
        check(H, t, d, keys)
    for part in np.array_split(np.arange(slots), 5):
        assert np.array_equal(t.erase(up(H, keys[part])).cpu().numpy(), d.erase(keys[part]))
        check(H, t, d, keys)
    assert t.size() == 0 and t.check() == 0
    t.close()


@pytest.mark.parametrize("n", [4_000_000, 4_000_001, 4_000_127])
@pytest.mark.parametrize("off", [0, 1, 4])
def test_long_find_batches(H, n, off):
    """Find batches long enough for four runs per warp and store, ragged ones
    and found flags at any byte offset: the same answers as in short batches."""
    t = H.HiveTable(1 << 16)
    keys, c = W.take_keys(31, 0, 50_000)
    vals = W.values_for(keys, 31)
    t.insert(up(H, keys), up(H, vals))
    pool = up(H, np.concatenate([keys, W.take_keys(31, c, 50_000)[0],
                                 np.array([0xFFFFFFFE, 0xFFFFFFFF], np.uint32)]))
    g = torch.Generator(device="cuda")
    g.manual_seed(n + off)
    at = torch.randint(0, pool.numel(), (n,), generator=g, device="cuda")
    v0, f0 = t.find(pool)  # a short batch
    vals_out = torch.full((n + off,), -1, dtype=torch.int32, device="cuda")
    found = torch.full((n + off + 64,), 7, dtype=torch.uint8, device="cuda")
    t.find(pool[at], vals_out=vals_out[off:], found=found[off:off + n])
    assert torch.equal(vals_out[off:], v0[at]) and torch.equal(found[off:off + n], f0[at])
    assert bool((found[:off] == 7).all()) and bool((found[off + n:] == 7).all())
    assert t.check() == 2  # the reserved keys
    t.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("buckets", [1, 2, 3, 64])
@pytest.mark.parametrize("n", [1, 33, 700])
def test_small_tables_with_32_bit_entries(H, layout, buckets, n):
    """The same edges on tables with 32-bit entries: a 16-bit map and a set."""
    from test_gpu_hive32 import check_image as check_image32

    n = min(n, buckets * 32)
    rng = np.random.default_rng(n)
    if layout == 0:
        every = rng.permutation(0xFFFE).astype(np.uint32)
        keys, absent = every[:n].copy(), every[n:2 * n].copy()
        vals = rng.integers(0, 1 << 16, n).astype(np.uint32)
    else:
        keys, c = W.take_keys(600 + n, 0, n)
        absent, _ = W.take_keys(600 + n, c, n)
        vals = np.zeros(n, np.uint32)
    t = H.Hive32Table(buckets * 32, layout)
    d = oracle.Dict()
    probe = np.concatenate([keys, absent])
    for _ in range(3):
        assert np.array_equal(t.insert(up(H, keys), up(H, vals)).cpu().numpy(),
                              d.insert(keys, vals))
        for phase in range(2):
            v, f = t.find(up(H, probe))
            ev, ef = d.find(probe)
            assert np.array_equal(f.cpu().numpy(), ef) and np.array_equal(H.to_host_u32(v), ev)
            check_image32(t, d)
            if phase == 0:
                er = keys[::2].copy()
                assert np.array_equal(t.erase(up(H, er)).cpu().numpy(), d.erase(er))
    assert t.check() == 0
    t.close()


@pytest.mark.parametrize("bs", [16, 32])
def test_bulk_inserts_stored_by_region(H, bs):
    """Tables beyond 256 MB of words take large inserts in two kernels: claims,
    then stores by region.  Ragged batches with new and present keys, reserved
    keys and a status array, on a table whose last region is a partial one;
    the same finds, sizes and image as the CPU dictionary's."""
    slots = (1 << 25) + (1 << 20) + 32 * 77
    n = slots // 8 + 4097  # two ops a line and a ragged tile
    t = H.HiveTable(slots, bucket_slots=bs)
    keys, c = W.take_keys(71, 0, n)
    vals = W.values_for(keys, 71)
    st = t.insert(up(H, keys), up(H, vals))
    assert bool((st == H.INSERTED).all())
    new, c = W.take_keys(71, c, n // 2)
    k2 = np.concatenate([keys[: n // 2], new, np.array([0xFFFFFFFF, 0xFFFFFFFE], np.uint32)])
    v2 = W.values_for(k2, 72)
    order = np.random.default_rng(3).permutation(k2.size)
    k2, v2 = k2[order], v2[order]
    st = t.insert(up(H, k2), up(H, v2)).cpu().numpy()
    want = np.where(order < n // 2, H.REPLACED, H.INSERTED)
    want[order >= k2.size - 2] = H.RESERVED_KEY
    assert np.array_equal(st, want)
    assert t.size() == n + n // 2 and t.check() == 2  # the reserved keys
    d = oracle.Dict()
    d.insert(keys, vals)
    d.insert(k2, v2)
    check(H, t, d, np.concatenate([keys[:100_000], new[:100_000],
                                   W.take_keys(71, c, 100_000)[0]]))
    t.close()


@pytest.mark.parametrize("bs", [16, 32])
@pytest.mark.parametrize("n", [200_001, (1 << 18) - 1])
def test_new_keys_wait_in_the_warp_queue(H, bs, n):
    """Mixed batches of several chunks per warp that claim in the bulk kernel:
    new keys wait in their warp's queue and claim 32 at a time, the last ones
    at the end; on one table and as ragged segments of a multi-table batch."""
    slots = 1 << 20
    rng = np.random.default_rng(n + bs)
    live, c = W.take_keys(81, 0, slots * 94 // 100)
    new, _ = W.take_keys(81, c, n // 3)
    ops, keys, vals = W.mixed_batch(rng, live, new, n // 3, n // 4, n - n // 3 - n // 4, seed=81)
    o, k, v = torch.from_numpy(ops).cuda(), up(H, keys), up(H, vals)
    d = oracle.Dict()
    d.insert(live, W.values_for(live, 81))
    ev, es = d.execute(ops, keys, vals)
    t = H.HiveTable(slots, bucket_slots=bs)
    t.insert(up(H, live), up(H, W.values_for(live, 81)))
    vo, st = t.execute(o, k, v)
    assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
    check(H, t, d, keys)
    t.close()
    # the same ops as segments on two tables, in cuts that end inside a chunk
    tabs = [H.HiveTable(slots, bucket_slots=bs) for _ in range(2)]
    for x in tabs:
        x.insert(up(H, live), up(H, W.values_for(live, 81)))
    cuts = [0, 1, 33, n // 2, n - 5, n]
    m = H.HiveMulti(tabs, max_segments=16, max_ops=4 * n)
    vo = torch.full((2, n), -1, dtype=torch.int32, device="cuda")
    st = torch.full((2, n), 9, dtype=torch.uint8, device="cuda")
    segs = [{"table": j, "ops": o[a:b].clone(), "keys": k[a:b].clone(), "vals": v[a:b].clone(),
             "vals_out": vo[j, a:b], "status": st[j, a:b]}
            for a, b in zip(cuts, cuts[1:]) for j in range(2)]
    m.execute(segs)
    for j in range(2):
        assert np.array_equal(st[j].cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo[j]), ev)
        check(H, tabs[j], d, keys)
    m.close()
    for x in tabs:
        assert x.check() == 0
        x.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("n", [200_001, 400_000])
def test_new_keys_wait_in_the_warp_queue_of_32_bit_entries(H, layout, n):
    """The same queue on tables with 32-bit entries, filled until some of the
    queued keys find both buckets full."""
    from test_gpu_hive32 import check_image as check_image32

    rng = np.random.default_rng(n + layout)
    if layout == 0:
        pool, slots, n_live, n_new = rng.permutation(0xFFFE).astype(np.uint32), 1 << 16, 50_000, 14_000
        vmask = 0xFFFF
    else:
        slots, n_live, n_new, vmask = 1 << 18, 240_000, 20_000, 0
        pool, _ = W.take_keys(91, 0, n_live + n_new)
    live, new = pool[:n_live], pool[n_live:n_live + n_new]
    lv = (W.values_for(live, 91) & vmask).astype(np.uint32)
    ops, keys, vals = W.mixed_batch(rng, live, new, n_new, 1_000, n - n_new - 1_000, seed=91)
    vals = (vals & vmask).astype(np.uint32)
    t = H.Hive32Table(slots, layout, stash_permille=50)
    d = oracle.Dict()
    t.insert(up(H, live), up(H, lv))
    d.insert(live, lv)
    before = t.stats()["overflowed"]
    vo, st = t.execute(torch.from_numpy(ops).cuda(), up(H, keys), up(H, vals))
    ev, es = d.execute(ops, keys, vals)
    assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
    if layout == 1:
        assert t.stats()["overflowed"] > before
    check_image32(t, d)
    assert t.check() == 0
    t.close()
