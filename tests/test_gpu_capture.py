"""Captured calls and the scratch arrays of eager ones: a replayed graph uses
nothing that a larger eager call frees."""
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


def test_captured_bulk_insert_survives_larger_eager_ones(H):
    """A table large enough for inserts by region: a captured insert, an eager
    one that needs a longer list, the graph replayed on new keys.  A slightly
    longer list costs no reallocation."""
    slots = (1 << 25) + (1 << 16)
    n = slots // 8 + 1000
    sizes = [n, n, n + 40_000, n, (1 << 23) + 5, n]  # eager, replay, eager, replay, eager, replay
    keys, _ = W.take_keys(611, 0, sum(sizes))
    vals = W.values_for(keys, 611)
    dk, dv = H.to_device_u32(keys), H.to_device_u32(vals)
    t = H.HiveTable(slots)
    parts, at = [], 0
    for m in sizes:
        parts.append((dk[at:at + m], dv[at:at + m]))
        at += m
    t.insert(*parts[0], status=None)
    gk, gv = torch.empty_like(dk[:n]), torch.empty_like(dv[:n])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        st = t.insert(gk, gv)
    mem = t.memory()
    for i in range(1, len(parts)):
        if i % 2:  # replay
            gk.copy_(parts[i][0])
            gv.copy_(parts[i][1])
            g.replay()
            assert bool((st == H.INSERTED).all())
        else:
            assert bool((t.insert(*parts[i]) == H.INSERTED).all())
            # the longer lists of the last one: 24 bytes an op and the tiles'
            # offsets, beside the ones that the graph uses
            new = 0 if i == 2 else (1 << 24) * 24 + (1 << 24) // 2048 * 129 * 2
            assert t.memory()[0] == mem[0] + new
    v, f = t.find(dk)
    assert bool((f == 1).all()) and bool((v == dv).all())
    assert t.size() == keys.size and t.check() == 0
    t.close()


@pytest.mark.parametrize("call", ["insert", "execute", "fused", "set_insert", "set_execute"])
def test_captured_small_calls_survive_larger_eager_ones(H, call):
    """The op lists of the update calls, on a table so full that keys go
    through them."""
    slots, n, big = 1 << 18, 512, 1 << 17
    n0 = slots * 45 // 100
    keys, _ = W.take_keys(621, 0, n0 + big + 2 * n)
    vals = np.zeros_like(keys) if call.startswith("set") else W.values_for(keys, 621)
    dk, dv = H.to_device_u32(keys), H.to_device_u32(vals)
    t = H.Hive32Table(slots, H.KEY_ONLY) if call.startswith("set") else H.HiveTable(slots)
    ops = torch.zeros(big, dtype=torch.uint8, device="cuda")

    def run(a, b):
        if call.endswith("insert"):
            return t.insert(dk[a:b], dv[a:b])
        kw = {"fused": True} if call == "fused" else {}
        return t.execute(ops[:b - a], dk[a:b], dv[a:b], **kw)[1]

    at = n0 + big
    for a in range(0, n0, 1 << 14):  # calls too small to lengthen the lists
        run(a, min(a + (1 << 14), n0))
    gk, gv = dk[at:at + n].clone(), dv[at:at + n].clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        if call.endswith("insert"):
            st = t.insert(gk, gv)
        else:
            kw = {"fused": True} if call == "fused" else {}
            st = t.execute(ops[:n], gk, gv, **kw)[1]
    mem = t.memory()[0] if isinstance(t, H.HiveTable) else 0
    assert bool((run(n0, n0 + big) == H.INSERTED).all())
    if mem:  # both lists of 2^16 entries stay beside the new ones
        assert t.memory()[0] == mem + 12 * big * (2 if call == "execute" else 1)
    for j in range(2):
        gk.copy_(dk[at + j * n:at + (j + 1) * n])
        gv.copy_(dv[at + j * n:at + (j + 1) * n])
        g.replay()
        assert bool((st == H.INSERTED).all())
    v, f = t.find(dk)
    assert bool((f == 1).all()) and bool((v == dv).all())
    assert t.size() == keys.size and t.check() == 0
    t.close()
