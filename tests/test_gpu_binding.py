"""The native call path of the Python binding against the Python one: the same
results, allocations and refusals, for every kind of argument a call takes."""
import numpy as np
import pytest

from paper_2510_15095_gb300 import workload as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Never:
    """A native module that leaves every call to the Python code."""

    def __getattr__(self, name):
        return lambda *a: NotImplemented


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15095_gb300 import hive
    hive.load_library()
    return hive


class Sub(torch.Tensor):
    pass


def outcome(f):
    try:
        r = f()
    except Exception as e:  # noqa: BLE001
        return type(e), str(e)
    r = r if isinstance(r, tuple) else (r,)
    return tuple(None if x is None else (x.dtype, tuple(x.shape), x.device, x.cpu().numpy().copy())
                 for x in r)


def same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        if isinstance(x, tuple) and len(x) == 4:
            assert x[:3] == y[:3] and np.array_equal(x[3], y[3])
        else:
            assert x == y


@pytest.mark.parametrize("kind", ["map", "set"])
def test_native_and_python_paths_agree(H, kind):
    keys, c = W.take_keys(3, 0, 1000)
    dk = H.to_device_u32(keys)
    dv = H.to_device_u32(W.values_for(keys, 3))
    ops = torch.from_numpy(np.tile(np.array([0, 1, 2, 1], np.uint8), 250)).cuda()
    side = torch.cuda.Stream()
    calls = [
        lambda t: t.insert(dk, dv), lambda t: t.insert(dk, dv, status=None),
        lambda t: t.insert(dk, dv, status=False),
        lambda t: t.insert(dk, dv, status=torch.empty(1000, dtype=torch.uint8, device="cuda")),
        lambda t: t.insert(dk.view(torch.uint32), dv), lambda t: t.insert(dk[::2], dv),
        lambda t: t.insert(dk, dv[:10]), lambda t: t.insert(dk.cpu(), dv),
        lambda t: t.insert(dk.long(), dv), lambda t: t.insert(dk, dv, status=dk),
        lambda t: t.find(dk), lambda t: t.find(dk, found=None), lambda t: t.find(dk, found=False),
        lambda t: t.find(dk[:0]), lambda t: t.find(dk[1:]), lambda t: t.find(dk.view(2, 500)),
        lambda t: t.find(dk, vals_out=torch.empty_like(dk)),
        lambda t: t.find(dk, vals_out=torch.empty(7, dtype=torch.int32, device="cuda")),
        lambda t: t.find(dk.as_subclass(Sub)), lambda t: t.find(dk.t()), lambda t: t.find(None),
        lambda t: t.find(dk, vals_out=True), lambda t: t.find(dk, stream=3),
        lambda t: t.find(dk, stream=torch.cuda.current_stream()),
        lambda t: (side.wait_stream(torch.cuda.current_stream()), t.find(dk, stream=side),
                   side.synchronize())[1],
        lambda t: t.execute(ops, dk, dv), lambda t: t.execute(ops, dk),
        lambda t: t.execute(ops[:9], dk, dv), lambda t: t.execute(ops, dk, None),
        lambda t: t.erase(dk[:100]), lambda t: t.erase(dk, status=None),
        lambda t: t.erase(dk, status=torch.empty(5, dtype=torch.uint8, device="cuda")),
    ]
    if kind == "map":
        make = lambda: H.HiveTable(1 << 12)  # noqa: E731
        calls += [lambda t: t.insert(dk, None), lambda t: t.insert_noalloc(dk, dv),
                  lambda t: t.execute(ops, dk, dv, fused=True)]
    else:
        make = lambda: H.Hive32Table(1 << 12, H.KEY_ONLY)  # noqa: E731
        calls += [lambda t: t.insert(dk)]
    a, b = make(), make()
    b._N = Never()
    for i, f in enumerate(calls):
        same(outcome(lambda: f(a)), outcome(lambda: f(b)))
        assert a.size() == b.size(), i
    a.close()
    b.close()
    same(outcome(lambda: a.find(dk)), outcome(lambda: b.find(dk)))  # closed: refused


@pytest.mark.parametrize("resizable", [False, True])
def test_multi_segments_native_and_python(H, resizable):
    rng = np.random.default_rng(1)
    got = []
    for native in (True, False):
        kw = dict(resizable=True, max_slots=1 << 14) if resizable else {}
        tabs = [H.HiveTable(1 << 10, bucket_slots=16, **kw) for _ in range(3)]
        m = H.HiveMulti(tabs, max_segments=8, max_ops=1 << 14)
        if not native:
            m._N = Never()
        rng = np.random.default_rng(1)
        res = []
        for step in range(3):
            segs = []
            for t in range(3 if step < 2 else 1):
                n = int(rng.integers(1, 300))
                keys, _ = W.take_keys(50 + t, 300 * step, n)
                dev = "cuda" if t != 1 else "cpu"
                mk = (lambda x: x.cuda()) if dev == "cuda" else (lambda x: x.pin_memory())
                segs.append({"table": t, "ops": mk(torch.zeros(n, dtype=torch.uint8)),
                             "keys": mk(torch.from_numpy(keys.view(np.int32).copy())),
                             "vals": mk(torch.ones(n, dtype=torch.int32)),
                             "status": mk(torch.full((n,), 9, dtype=torch.uint8))})
                if t == 2:
                    segs[-1]["n_insert"] = n
            m.execute(segs)
            sizes = m.bounds()
            torch.cuda.synchronize()
            assert sizes == [t.size() for t in tabs]
            res += [s["status"].cpu().numpy().copy() for s in segs] + [np.array(sizes)]
        bad = {"table": 0, "ops": segs[0]["ops"], "keys": segs[0]["keys"].long()}
        for segs_bad in ([bad], [{"table": 9, **{k: segs[0][k] for k in ("ops", "keys")}}],
                         [{"ops": segs[0]["ops"], "keys": segs[0]["keys"]}]):
            with pytest.raises(Exception) as e:
                m.execute(segs_bad)
            res.append((type(e.value), str(e.value)))
        got.append(res)
        m.close()
        for t in tabs:
            t.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y
