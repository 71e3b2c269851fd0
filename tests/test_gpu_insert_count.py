"""Growth of a resizable table before a mixed batch follows the batch's exact
number of inserts: counted 16 op codes at a time, at any alignment of the op
array and for ragged lengths, and not counted when even n new keys would not
grow the table.  The capacity after each call equals the policy model's."""
import numpy as np
import pytest

import oracle
from paper_2510_15095_gb300 import workload as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1, 15])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 4097])
def test_capacity_follows_the_insert_count(off, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15095_gb300 import hive as H
    rng = np.random.default_rng(n * 16 + off)
    t = H.HiveTable(64, max_slots=1 << 16, resizable=True, resize_batch=1, bucket_slots=16)
    pol = oracle.Policy(4, (1 << 16) // 16, S=16, K=1)
    d = oracle.Dict()
    live, c = np.zeros(0, np.uint32), 0
    for b in range(6):
        n_ins = int(rng.integers(0, n + 1))
        n_er = min(int(rng.integers(0, n - n_ins + 1)), live.size)
        new, c = W.take_keys(41, c, n)
        ops, keys, vals = W.mixed_batch(rng, live, new, n_ins, n_er, n - n_ins - n_er, seed=b)
        if ops.size == 0:
            continue
        pad = torch.zeros(ops.size + off, dtype=torch.uint8, device="cuda")  # zeros read as inserts
        pad[off:] = torch.from_numpy(ops).cuda()
        pol.grow(len(d), int((ops == 0).sum()))
        vo, st = t.execute(pad[off:], H.to_device_u32(keys), H.to_device_u32(vals))
        ev, es = d.execute(ops, keys, vals)
        pol.shrink(len(d))
        assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
        assert t.capacity() == 16 * pol.state[0]
        assert t.size() == len(d)
        live, _ = d.dump()
    assert t.check() == 0
    t.close()
