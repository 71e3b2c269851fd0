"""Probes that stage whole buckets (tables of 32-slot buckets created with a
stage_wait_limit that is not reached): several rounds per warp, hits in either
bucket, claims without tags at hand, against the oracle."""
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


@pytest.mark.parametrize("resizable", [False, True])
@pytest.mark.parametrize("n_mixed", [33, 5_000, (1 << 18) + 77])  # claims at once, or in their own kernel
def test_staged_rounds_that_complete(H, n_mixed, resizable):
    slots = 1 << 19
    kw = dict(resizable=True, max_slots=slots * 4) if resizable else {}
    t = H.HiveTable(slots, bucket_slots=32, stage_wait_limit=1 << 22, **kw)
    d = oracle.Dict()
    up = H.to_device_u32
    keys, c = W.take_keys(801, 0, slots * 9 // 10)
    vals = W.values_for(keys, 801)
    assert np.array_equal(t.insert(up(keys), up(vals)).cpu().numpy(), d.insert(keys, vals))
    rng = np.random.default_rng(n_mixed)
    live, _ = d.dump()
    new, c = W.take_keys(801, c, n_mixed // 4)
    ops, mk, mv = W.mixed_batch(rng, live, new, new.size, n_mixed // 4,
                                n_mixed - new.size - n_mixed // 4, seed=801)
    vo, st = t.execute(torch.from_numpy(ops).cuda(), up(mk), up(mv))
    ev, es = d.execute(ops, mk, mv)
    assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
    part = keys[::3]  # replaced where they are, inserted where the batch erased them
    assert np.array_equal(t.insert(up(part), up(part)).cpu().numpy(), d.insert(part, part))
    absent, _ = W.take_keys(801, c, 100_001)
    gone = np.concatenate([keys[1::5], absent[:1000]])
    assert np.array_equal(t.erase(up(gone)).cpu().numpy(), d.erase(gone))
    q = np.concatenate([keys, new, absent])
    v, f = t.find(up(q))
    ev, ef = d.find(q)
    assert np.array_equal(H.to_host_u32(v), ev) and np.array_equal(f.cpu().numpy(), ef)
    img = t.dump()
    code, where = oracle.check_image(img, img["S"], d, None)
    assert code == 0, f"invariant {code} fails at {where}"
    assert t.check() == 0  # no wait gave up
    t.close()
