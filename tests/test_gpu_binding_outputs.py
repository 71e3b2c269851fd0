"""Outputs of the native call path: written through the tensor's own storage,
and the error of an output that cannot be allocated."""
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


@pytest.mark.parametrize("call", ["find", "insert", "erase", "multi"])
def test_copy_on_write_outputs_get_their_own_storage(H, call):
    """An output that shares its storage with another tensor until it is
    written (a lazy clone) must not write into that tensor."""
    n = 512
    keys, _ = W.take_keys(31, 0, n)
    vals = W.values_for(keys, 31)
    dk, dv = H.to_device_u32(keys), H.to_device_u32(vals)
    words = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    flags = torch.full((n,), 77, dtype=torch.uint8, device="cuda")
    out, st = torch._lazy_clone(words), torch._lazy_clone(flags)
    t = H.HiveTable(1 << 11)
    if call != "insert":
        t.insert(dk, dv)
    if call == "find":
        t.find(dk, vals_out=out, found=st)
        assert np.array_equal(H.to_host_u32(out), vals) and bool((st == 1).all())
    elif call == "insert":
        t.insert(dk, dv, status=st)
        assert bool((st != 77).all())
    elif call == "erase":
        t.erase(dk, status=st)
        assert bool((st != 77).all()) and t.size() == 0
    else:
        m = H.HiveMulti([t], max_segments=1, max_ops=n)
        ops = torch.full((n,), H.OP_FIND, dtype=torch.uint8, device="cuda")
        m.execute([{"table": 0, "ops": ops, "keys": dk, "vals_out": out, "status": st}])
        torch.cuda.synchronize()
        assert np.array_equal(H.to_host_u32(out), vals) and bool((st != 77).all())
        m.close()
    assert bool((words == -7).all()) and bool((flags == 77).all())
    t.close()


@pytest.mark.parametrize("call", ["find", "insert", "erase", "execute"])
def test_output_that_cannot_be_allocated(H, call):
    """torch.OutOfMemoryError, as from torch.empty, and the table untouched."""
    n = 1 << 24
    t = H.HiveTable(1 << 12)
    dk = torch.arange(n, dtype=torch.int32, device="cuda")
    ops = torch.zeros(n, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    dev = torch.cuda.current_device()
    total = torch.cuda.get_device_properties(dev).total_memory
    # 1 MB is left to PyTorch's allocator: an output takes 16 MB or 64
    torch.cuda.set_per_process_memory_fraction(
        (torch.cuda.memory_reserved(dev) + (1 << 20)) / total, dev)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            {"find": lambda: t.find(dk), "insert": lambda: t.insert(dk, dk),
             "erase": lambda: t.erase(dk), "execute": lambda: t.execute(ops, dk, dk)}[call]()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0, dev)
    assert t.size() == 0 and t.check() == 0
    t.close()
