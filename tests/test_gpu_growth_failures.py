"""Growth that cannot get memory (the failure is made on the host): the call
returns OOM, the table keeps its capacity and every key, and the same call
succeeds once memory can be had."""
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
    yield hive
    hive.debug_fail_alloc(0)


def up(H, a):
    return H.to_device_u32(a)


def check(H, t, d, keys):
    v, f = t.find(up(H, keys))
    ev, ef = d.find(keys)
    assert np.array_equal(H.to_host_u32(v), ev) and np.array_equal(f.cpu().numpy(), ef)
    img = t.dump()
    code, where = oracle.check_image(img, img["S"], d, None)
    assert code == 0, f"invariant {code} fails at {where}"
    assert t.size() == len(d)


def on_demand(H, bs, **kw):
    # 2^18 slots fill the 2 MB that the driver maps at a time
    return H.HiveTable(1 << 18, max_slots=1 << 22, resizable=True, bucket_slots=bs,
                       map_on_demand=True, **kw)


@pytest.mark.parametrize("bs", [16, 32])
def test_reserve_without_memory(H, bs):
    t, d = on_demand(H, bs), oracle.Dict()
    keys, _ = W.take_keys(701, 0, 100_000)
    vals = W.values_for(keys, 701)
    t.insert(up(H, keys), up(H, vals))
    d.insert(keys, vals)
    cap = t.capacity()
    H.debug_fail_alloc(1)
    with pytest.raises(H.HiveError) as e:
        t.reserve(1 << 20)
    assert "OOM" in str(e.value) and t.capacity() == cap and t.stats()["splits"] == 0
    check(H, t, d, keys)
    t.reserve(1 << 20)
    assert t.capacity() >= 1 << 20
    check(H, t, d, keys)
    assert t.check() == 0
    t.close()


@pytest.mark.parametrize("asynchronous", [False, True])
def test_multi_table_growth_without_memory(H, asynchronous):
    tabs = [on_demand(H, 16) for _ in range(3)]
    dicts = [oracle.Dict() for _ in tabs]
    m = H.HiveMulti(tabs, max_segments=4, max_ops=1 << 20, asynchronous=asynchronous)
    keys, vals, segs = [], [], []
    for j in range(3):
        k, _ = W.take_keys(710 + j, 0, 300_000)
        keys.append(k)
        vals.append(W.values_for(k, 710 + j))
        segs.append({"table": j, "ops": torch.zeros(k.size, dtype=torch.uint8, device="cuda"),
                     "keys": up(H, k), "vals": up(H, vals[j]),
                     "status": torch.full((k.size,), 9, dtype=torch.uint8, device="cuda")})
    caps = [t.capacity() for t in tabs]
    H.debug_fail_alloc(2)  # the second table's buckets
    with pytest.raises(H.HiveError) as e:
        m.execute(segs)
    assert "OOM" in str(e.value)
    torch.cuda.synchronize()
    assert [t.capacity() for t in tabs] == caps and [t.size() for t in tabs] == [0, 0, 0]
    m.execute(segs)
    torch.cuda.synchronize()
    for j, t in enumerate(tabs):
        assert np.array_equal(segs[j]["status"].cpu().numpy(), dicts[j].insert(keys[j], vals[j]))
        assert t.capacity() > caps[j]
        check(H, t, dicts[j], keys[j])
        assert t.check() == 0
    m.close()
    for t in tabs:
        t.close()


@pytest.mark.parametrize("bs", [16, 32])
@pytest.mark.parametrize("call", ["insert", "execute", "execute_large", "fused"])
def test_batch_that_cannot_grow_in_the_middle(H, bs, call):
    """Inserts that fill the last slots find no room, and the table cannot get
    memory for the split they ask for: every other op of the batch has run, the
    op lists start empty in the next call, and the same inserts succeed then."""
    slots = 1 << 18
    n_new = 60_000
    keys, c = W.take_keys(721, 0, slots)
    live, new = keys[:slots - n_new], keys[slots - n_new:]
    t = on_demand(H, bs, grow=(1, 1), shrink=(1, 10), max_evictions=1, stash_permille=0)
    d = oracle.Dict()
    lv = W.values_for(live, 721)
    for part in np.array_split(np.arange(live.size), 2):
        t.insert(up(H, live[part]), up(H, lv[part]))
    d.insert(live, lv)
    n_find = {"insert": 0, "execute": 100_000, "execute_large": 300_000, "fused": 100_000}[call]
    rng = np.random.default_rng(bs)
    mk = np.concatenate([new, rng.choice(live, n_find)])
    ops = np.concatenate([np.zeros(n_new, np.uint8), np.ones(n_find, np.uint8)])
    order = rng.permutation(mk.size)
    mk, ops = mk[order], ops[order]
    mv = np.where(ops == 0, W.values_for(mk, 722), 0).astype(np.uint32)
    args = (torch.from_numpy(ops).cuda(), up(H, mk), up(H, mv))

    def run():
        if call == "insert":
            return t.insert(args[1], args[2])
        return t.execute(*args, fused=call == "fused")[1]

    cap = t.capacity()
    if call.startswith("execute") or call == "fused":  # the lists have the batch's length
        t.execute(torch.ones_like(args[0]), args[1])
    else:
        t.erase(args[1])  # absent
        t.execute(torch.ones_like(args[0]), args[1])
    H.debug_fail_alloc(1)
    with pytest.raises(H.HiveError) as e:
        run()
    assert "OOM" in str(e.value) and t.capacity() == cap
    d.execute(ops, mk, mv)
    there = t.find(up(H, new))[1].cpu().numpy().astype(bool)
    assert 0 < (~there).sum() < n_new
    d.erase(new[~there])
    check(H, t, d, keys)
    assert t.check() == 4  # FULL: inserts found no room
    st = run()
    assert np.array_equal(st.cpu().numpy(), d.execute(ops, mk, mv)[1])
    assert t.capacity() > cap
    check(H, t, d, keys)
    assert t.check() == 0
    t.close()


@pytest.mark.parametrize("bs", [16, 32])
def test_slot_tags_are_mapped_on_demand(H, bs):
    """A large max_slots costs address space, not memory, beyond 12 bytes a
    bucket; and a table whose tags cannot be mapped when its buckets can."""
    nb_max = 1 << 26
    t = H.HiveTable(1 << 16, max_slots=nb_max * bs, resizable=True, bucket_slots=bs,
                    map_on_demand=True, stash_permille=0)
    committed, reserved = t.memory()
    assert committed < 12 * nb_max + (16 << 20) and reserved >= 9 * bs * nb_max
    t.close()
    # 2^21 slots: 16 MB of words and 2 MB of tags are mapped, both full
    t, d = on_demand(H, bs), oracle.Dict()
    t.reserve(1 << 21)
    keys, c = W.take_keys(731, 0, 1 << 20)
    vals = W.values_for(keys, 731)
    t.insert(up(H, keys), up(H, vals))
    d.insert(keys, vals)
    assert t.capacity() == 1 << 21
    H.debug_fail_alloc(2)  # the words' mapping succeeds, the tags' fails
    with pytest.raises(H.HiveError) as e:
        t.reserve((1 << 21) + 1)
    assert "OOM" in str(e.value) and t.capacity() == 1 << 21
    check(H, t, d, keys)
    more, _ = W.take_keys(731, c, 1 << 21)
    mv = W.values_for(more, 731)
    assert np.array_equal(t.insert(up(H, more), up(H, mv)).cpu().numpy(), d.insert(more, mv))
    assert t.capacity() > 1 << 21
    check(H, t, d, np.concatenate([keys, more]))
    # shrink gives the memory back, growth finds it filled anew
    c0 = t.memory()[0]
    gone = np.concatenate([keys, more])[: 3 * (1 << 20) - 50_000]
    assert np.array_equal(t.erase(up(H, gone)).cpu().numpy(), d.erase(gone))
    assert t.memory()[0] < c0 - (16 << 20)
    check(H, t, d, keys)
    t.insert(up(H, gone), up(H, W.values_for(gone, 732)))
    d.insert(gone, W.values_for(gone, 732))
    check(H, t, d, gone)
    assert t.check() == 0
    t.close()
