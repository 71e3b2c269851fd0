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
