"""The kernels of one call as a chain of dependent launches: the same results
when calls follow one another without a wait, on a side stream, and when a
chain is captured into a CUDA graph and replayed on new inputs."""
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


def batches(seed, slots, n, count):
    rng = np.random.default_rng(seed)
    live, c = W.take_keys(seed, 0, slots * 93 // 100)
    first, d, out = live, oracle.Dict(), []
    d.insert(live, W.values_for(live, seed))
    for b in range(count):
        new, c = W.take_keys(seed, c, n // 4)
        ops, keys, vals = W.mixed_batch(rng, live, new, n // 4, n // 4, n // 2, seed=b)
        out.append((ops, keys, vals, *d.execute(ops, keys, vals)))
        live, _ = d.dump()
    return first, d, out


def check_end(t, d):
    img = t.dump()
    code, where = oracle.check_image(img, img["S"], d, None)
    assert code == 0, f"invariant {code} fails at {where}"
    assert t.check() == 0


@pytest.mark.parametrize("bs", [16, 32])
@pytest.mark.parametrize("n", [64, 4096, 1 << 18])
def test_calls_back_to_back_and_replayed(H, bs, n):
    slots = max(1 << 13, 4 * n)
    first, d, todo = batches(n + bs, slots, n, 6)
    t = H.HiveTable(slots, bucket_slots=bs)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        t.insert(H.to_device_u32(first), H.to_device_u32(W.values_for(first, n + bs)), status=None)
        up = [(torch.from_numpy(o).cuda(), H.to_device_u32(k), H.to_device_u32(v))
              for o, k, v, _, _ in todo]
        got = [t.execute(*x) for x in up[:3]]  # no wait between the calls
        side.synchronize()
        # one captured chain, replayed on three more batches
        ops, keys, vals = (x.clone() for x in up[3])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            vo, st = t.execute(ops, keys, vals)
        for x in up[3:]:
            for dst, src in zip((ops, keys, vals), x):
                dst.copy_(src)
            g.replay()
            got.append((vo.clone(), st.clone()))
        side.synchronize()
    for (vo, st), (_, _, _, ev, es) in zip(got, todo):
        assert np.array_equal(st.cpu().numpy(), es) and np.array_equal(H.to_host_u32(vo), ev)
    check_end(t, d)
    t.close()
