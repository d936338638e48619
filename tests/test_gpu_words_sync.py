"""The producer warp of the sweep over fixed-point words on the GPU: what its
lanes agree on before one of them acts for all, bit for bit against the CPU
oracle."""
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


# every lane watches another tile's step counter (up to 19 in the tile's record,
# more of them in the list), one plane or row to a tile, so that each step
# hangs on tiles that other SMs finished just before
@pytest.mark.parametrize("dims,kw", [
    ((48, 40, 36), dict(split=(4, 5, 3), tile_y=2, tile_z=1)),
    ((260, 128, 9), dict(cuts=([0, 4, 260], [0, 128], [0, 3, 9]))),
    ((64, 64, 64), dict(split=(2, 2, 2), threads=256, cells_per_thread=1)),
])
def test_dependencies_watched_by_different_lanes(od, dims, kw):
    want = oracle.solve(*dims, 11, 1, 150)
    with od.Jacobi3D(*dims, seed=11, path="persistent", **kw) as s:
        s.step(150)
        assert same(s.read(), want)


# a wait that runs out ends every warp of every CTA with the error recorded,
# whatever the shape, and leaves the GPU to the next context
@pytest.mark.parametrize("kw", [dict(threads=128, cells_per_thread=2), dict(threads=128, cells_per_thread=4),
                                dict(threads=256, cells_per_thread=4), dict(threads=512, cells_per_thread=1)])
@pytest.mark.parametrize("tile", [0, 5])
def test_a_wait_that_runs_out_ends_the_launch(od, kw, tile):
    with od.Jacobi3D(48, 40, 32, split=(2, 2, 2), seed=1, path="persistent", tile_z=4, spin_limit_ns=100_000_000,
                     **kw) as s:
        s.stall_tile(tile)
        s.step(20)
        with pytest.raises(od.ODError) as ei:
            s.sync()
        assert ei.value.status == od._native.OD_ETIMEOUT
    want = oracle.solve(48, 40, 32, 1, 1, 20)
    with od.Jacobi3D(48, 40, 32, split=(2, 2, 2), seed=1, path="persistent", tile_z=4, **kw) as s:
        s.step(20)
        assert same(s.read(), want)


# a wait limit too short for any copy: the launch ends with the error (or beats
# the limit), its copies landed, and CTAs of other contexts, which take over the
# shared memory, compute what they should
@pytest.mark.parametrize("arith", [-1, 2])
@pytest.mark.parametrize("path", ["persistent", "fused", "per_chare"])
def test_copies_in_flight_land_before_a_cta_gives_up(od, path, arith):
    dims = (256, 64, 48)
    want = oracle.solve(*dims, 2, 1, 12)
    with od.Jacobi3D(*dims, split=(2, 2, 2), seed=2, path=path, arith=arith) as good:
        with od.Jacobi3D(*dims, split=(2, 2, 2), seed=2, path=path, arith=arith, spin_limit_ns=1) as s:
            for _ in range(4):
                good.step(3)
                try:
                    s.step(3)
                    s.sync()
                except od.ODError as e:
                    assert e.status in (od._native.OD_ETIMEOUT, od._native.OD_ESTATE)
        assert same(good.read(), want)


# limits as good as none, whose multiples by 2 and 4 pass the end of 64 bits
@pytest.mark.parametrize("limit", [1 << 61, 1 << 62, (1 << 62) + 1, 1 << 63, (1 << 64) - 1])
def test_wait_limits_of_any_size(od, limit):
    want = oracle.solve(64, 64, 64, 7, 1, 40)
    with od.Jacobi3D(64, 64, 64, split=(2, 2, 2), seed=7, path="persistent", spin_limit_ns=limit) as s:
        s.step(40)
        assert same(s.read(), want)


# rows of 500 cells in 256 x 2: the default ring fills the shared memory of
# three CTAs an SM to within a kilobyte
def test_resident_ctas_of_two_cells_a_thread(od):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with od.Jacobi3D(500, 64, 64, split=(1, 1, 1), seed=2, path="persistent", threads=256, cells_per_thread=2,
                     tile_z=4) as s:
        s.step(3)
        assert same(s.read(), oracle.solve(500, 64, 64, 2, 1, 3))
        assert s.stats()["persistent_grid"] == 3 * sms
