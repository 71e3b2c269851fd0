"""Synchronous groups of fixed tables: a batch is not waited for, and nothing
that its caller can see depends on that."""
import numpy as np
import pytest

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


def seg(H, table, keys, dev="cuda", op=0):
    to = (lambda x: x.cuda()) if dev == "cuda" else (lambda x: x.pin_memory())
    n = keys.size
    return {"table": table, "ops": to(torch.full((n,), op, dtype=torch.uint8)),
            "keys": to(torch.from_numpy(keys.view(np.int32).copy())),
            "vals": to(torch.from_numpy(W.values_for(keys, 5).view(np.int32).copy())),
            "vals_out": to(torch.full((n,), -3, dtype=torch.int32)),
            "status": to(torch.full((n,), 9, dtype=torch.uint8))}


def test_bounds_follow_the_newest_size(H):
    """hive_multi_bounds after the tables were cleared, after another group's
    batch on the same tables, and with a group closed before its sizes were
    taken."""
    keys, _ = W.take_keys(5, 0, 1000)
    tabs = [H.HiveTable(1 << 12, bucket_slots=16) for _ in range(2)]
    a = H.HiveMulti(tabs, max_segments=4, max_ops=1 << 12)
    b = H.HiveMulti(tabs[::-1], max_segments=4, max_ops=1 << 12)
    a.execute([seg(H, 0, keys[:100]), seg(H, 1, keys[:40])])
    tabs[0].clear()
    assert a.bounds() == [0, 40] and b.bounds() == [40, 0]
    a.execute([seg(H, 0, keys[:100])])
    b.execute([seg(H, 1, keys[100:130]), seg(H, 0, keys[500:507])])
    assert a.bounds() == [130, 47]
    a.execute([seg(H, 0, keys[200:300])])
    c = H.HiveMulti(tabs, max_segments=4, max_ops=1 << 12, asynchronous=True)
    assert c.bounds() == [230, 47]
    c.close()
    a.execute([seg(H, 1, keys[300:310])])
    a.close()
    assert b.bounds() == [57, 230]
    b.execute([seg(H, 0, keys[400:401])])
    tabs[1].close()  # a table and the group in either order
    b.close()
    assert tabs[0].size() == 230
    tabs[0].close()


def test_batches_on_two_streams_run_in_order(H):
    """Consecutive batches of a group on different streams, none of them waited
    for: each one's finds see the batch before."""
    n, rounds = 150_000, 12
    keys, _ = W.take_keys(6, 0, n * rounds)
    tabs = [H.HiveTable(1 << 21, bucket_slots=16) for _ in range(2)]
    m = H.HiveMulti(tabs, max_segments=4, max_ops=4 * n)
    streams = [torch.cuda.Stream() for _ in range(2)]
    batches = []
    for r in range(rounds):
        part = keys[n * r:n * (r + 1)]
        segs = [seg(H, 0, part), seg(H, 1, part)]
        if r:
            prev = keys[n * (r - 1):n * r]
            segs += [seg(H, 0, prev, op=H.OP_FIND), seg(H, 1, prev, op=H.OP_FIND)]
        batches.append(segs)
    torch.cuda.synchronize()
    for r, segs in enumerate(batches):
        m.execute(segs, stream=streams[r % 2])
    assert m.bounds() == [n * rounds, n * rounds]
    torch.cuda.synchronize()
    for segs in batches:
        for s in segs[:2]:
            assert bool((s["status"] == H.INSERTED).all())
        for s in segs[2:]:
            assert bool((s["status"] == H.FOUND).all()) and bool((s["vals_out"] == s["vals"]).all())
    m.close()
    for t in tabs:
        assert t.check() == 0
        t.close()


@pytest.mark.parametrize("late", ["find", "size", "insert", "noalloc", "execute", "erase", "stats",
                                  "dump", "clear", "group"])
def test_single_calls_on_another_stream_follow_the_batch(H, late):
    """A batch that is still queued on a side stream, and a call on one of its
    tables on the current stream right after it."""
    n = 50_000
    keys, _ = W.take_keys(10, 0, n)
    t = H.HiveTable(1 << 17, bucket_slots=16)
    m = H.HiveMulti([t], max_segments=1, max_ops=n)
    other = H.HiveMulti([t], max_segments=1, max_ops=n)
    s, f = seg(H, 0, keys), seg(H, 0, keys, op=H.OP_FIND)
    dk, dv = s["keys"].clone(), s["vals"].clone()
    t.insert(dk, dv)  # scratch has its size
    t.execute(f["ops"], dk, dv)
    t.clear()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
    m.execute([s], stream=side)
    if late == "find":
        v, found = t.find(dk)
        assert bool((found == 1).all()) and bool((v == dv).all())
    elif late == "size":
        assert t.size() == n
    elif late in ("insert", "noalloc"):
        st = (t.insert if late == "insert" else t.insert_noalloc)(dk, dv)
        assert bool((st == H.REPLACED).all())
    elif late == "execute":
        assert bool((t.execute(f["ops"], dk, dv)[1] == H.FOUND).all())
    elif late == "erase":
        assert bool((t.erase(dk) == H.ERASED).all())
    elif late == "stats":
        assert t.stats()["claimed_fast"] >= n
    elif late == "dump":
        assert t.dump()["size"] == n
    elif late == "clear":
        t.clear()
        assert t.size() == 0 and m.bounds() == [0]
    else:
        other.execute([f])
        torch.cuda.current_stream().synchronize()
        assert bool((f["status"] == H.FOUND).all())
    torch.cuda.synchronize()
    assert bool((s["status"] == H.INSERTED).all())
    assert t.check() == 0
    for x in (m, other, t):
        x.close()


def test_capture_is_refused(H):
    """A captured batch would replay descriptors that later batches replace."""
    keys, _ = W.take_keys(7, 0, 100)
    t = H.HiveTable(1 << 12, bucket_slots=16)
    m = H.HiveMulti([t], max_segments=1, max_ops=1 << 10)
    s = seg(H, 0, keys)
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(H.HiveError) as e:
            m.execute([s])
        x += 1
    assert "CUDA" in str(e.value)
    g.replay()
    m.execute([s])
    assert m.bounds() == [100] and bool((x == 1).all())
    assert bool((s["status"] == H.INSERTED).all())
    m.close()
    t.close()


@pytest.mark.parametrize("native", [True, False])
def test_host_arrays_are_done_when_the_call_returns(H, native):
    """Results in pinned memory are read, and pinned inputs dropped and their
    memory handed out again, right after execute()."""
    n = 400_000
    keys, _ = W.take_keys(8, 0, 4 * n)
    t = H.HiveTable(1 << 22, bucket_slots=16)
    m = H.HiveMulti([t], max_segments=2, max_ops=2 * n)
    if not native:
        m._N = type("Never", (), {"multi": lambda *a: NotImplemented})()
    for r in range(4):
        s = seg(H, 0, keys[n * r:n * (r + 1)], dev="cpu")
        m.execute([s])
        status, want = s["status"].numpy().copy(), s["vals"].numpy().copy()
        assert (status == H.INSERTED).all()
        del s
        junk = [torch.full((n,), 1, dtype=torch.int32).pin_memory() for _ in range(4)]
        f = seg(H, 0, keys[n * r:n * (r + 1)], dev="cpu", op=H.OP_FIND)
        m.execute([f])
        assert (f["vals_out"].numpy() == want).all() and (f["status"].numpy() == H.FOUND).all()
        del f, junk
    assert m.bounds() == [4 * n]
    m.close()
    t.close()


@pytest.mark.parametrize("native", [True, False])
def test_arrays_live_as_long_as_their_batch(H, native):
    """Temporaries of the current stream in a batch that waits on another one."""
    n = 100_000
    keys, _ = W.take_keys(9, 0, 2 * n)
    t = H.HiveTable(1 << 19, bucket_slots=16)
    m = H.HiveMulti([t], max_segments=2, max_ops=2 * n)
    if not native:
        m._N = type("Never", (), {"multi": lambda *a: NotImplemented})()
    side = torch.cuda.Stream()
    warm = seg(H, 0, keys[:1])
    torch.cuda.synchronize()
    m.execute([warm], stream=side)
    for r in range(2):
        s = seg(H, 0, keys[n * r:n * (r + 1)])
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # about 0.1 s
        m.execute([s], stream=side)
        del s
        junk = [torch.full((n,), 7, dtype=torch.int32, device="cuda") for _ in range(4)]
        junk += [torch.full((n,), 2, dtype=torch.uint8, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        assert all(bool((x == x[0]).all()) for x in junk)
        del junk
    v, f = t.find(H.to_device_u32(keys))
    assert bool((f == 1).all()) and np.array_equal(H.to_host_u32(v), W.values_for(keys, 5))
    assert m.bounds() == [2 * n] and m._arrays == [[], []]
    m.close()
    t.close()
