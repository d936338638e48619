"""od_read beside a pending asynchronous export and after a failed launch."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def od():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_12734_gb300 import build
    build.build()
    import paper_2605_12734_gb300 as pkg
    return pkg


def same(got, want):
    return np.array_equal(np.ascontiguousarray(got).view(np.uint64), np.ascontiguousarray(want).view(np.uint64))


# the export of an older field may still be on its way to the buffer when the
# newer field is read into it: as pinned memory, which the gather writes in
# place, and by the address that the device has for it
@pytest.mark.parametrize("how", ["pinned", "address"])
def test_read_into_the_buffer_of_a_pending_export(od, how):
    import torch
    n = 200
    want = oracle.solve(n, n, n, 3, 1, 2)
    buf = torch.empty(n ** 3, dtype=torch.float64, pin_memory=True)
    with od.Jacobi3D(n, n, n, split=(2, 2, 2), seed=3, path="persistent") as s:
        s.step(1)
        s.read_async(buf)
        s.step(1)
        if how == "pinned":
            s.read(buf.numpy())
        else:
            od._native.check(od.lib().od_read(s._h, buf.data_ptr(), 1), "od_read")
        first = buf.numpy().copy()
        s.sync()
        assert same(first, want)
        assert same(buf.numpy(), want)


# a read that reports the error of a launch that gave up leaves dst alone
@pytest.mark.parametrize("where", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("arith", [-1, 12, 2])
def test_read_of_a_failed_context_leaves_dst(od, where, arith):
    import torch
    n = 48
    if where == "device":
        dst = torch.full((n ** 3,), -3.0, dtype=torch.float64, device="cuda:0")
    else:
        dst = torch.full((n ** 3,), -3.0, dtype=torch.float64, pin_memory=where == "pinned").numpy()
    with od.Jacobi3D(n, n, n, split=(2, 2, 2), seed=1, path="persistent", arith=arith,
                     spin_limit_ns=100_000_000) as s:
        s.stall_tile(0)
        s.step(3)
        for _ in range(2):
            with pytest.raises(od.ODError) as ei:
                s.read(dst)
            assert ei.value.status == od._native.OD_ETIMEOUT
            assert bool((dst == -3.0).all())
