"""The sweep over fixed-point field words on the GPU where its formats and its
schedule have edges, bit for bit against the CPU oracle: fields that leave,
straddle or outgrow the window, an import that changes the format of a running
context, faces fed from outside, and tiles with long dependency lists, one
plane, one row or deep rings."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

PATHS = ["persistent", "fused", "fused_graph", "per_chare", "graph"]


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


def field(kind, n, rng):
    u = rng.random(n)
    if kind == "edges":  # the window's ends, one step inside and outside of them, and powers of two
        ends = [1.0, np.nextafter(1.0, 0), np.nextafter(1.0, 2), 2.0 ** -8, np.nextafter(2.0 ** -8, 0),
                np.nextafter(2.0 ** -8, 1), 0.5, 0.25, 2.0 ** -7]
        return rng.choice(ends, n)
    if kind == "tiny":   # window values among ones far below it, zeros of both signs and subnormals
        v = np.where(u < 0.5, u, np.exp2(-rng.integers(9, 1070, n).astype(np.float64)))
        v[::5] = 0.0
        v[1::17] = -0.0
        v[2::23] = 5e-324
        return v
    if kind == "huge":   # near the top of the double range, some sums overflow
        return u * 1.5e308
    if kind == "infinite":
        u[::97] = np.inf
        return u
    return u


def solve_from(nx, ny, nz, seed, interior, iters):
    if nz == 0:
        P = oracle.init_padded_2d(nx, ny, seed, 1)
        P[1:-1, 1:-1] = interior.reshape(ny, nx)
        return oracle.sweep_2d(P, iters)[1:-1, 1:-1].ravel()
    P = oracle.init_padded(nx, ny, nz, seed, 1)
    P[1:-1, 1:-1, 1:-1] = interior.reshape(nz, ny, nx)
    return oracle.interior(oracle.sweep(P, iters))


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("kind", ["edges", "tiny", "huge", "infinite"])
def test_fields_outside_the_window(od, path, kind):
    nx, ny, nz, seed, iters = 37, 30, 26, 5, 6
    u = field(kind, nx * ny * nz, np.random.default_rng(len(kind)))
    want = solve_from(nx, ny, nz, seed, u, iters)
    with od.Jacobi3D(nx, ny, nz, split=(2, 3, 2), seed=seed, path=path) as s:
        s.write(u)
        s.step(iters)
        assert same(s.read(), want)
        probe = np.array([0, 1, nx, nx * ny - 1, nx * ny * nz - 1, 4321])
        assert same(s.read_cells(probe), want[probe])


@pytest.mark.parametrize("path", PATHS)
def test_import_that_changes_the_format(od, path):
    # each field's largest value asks for another window than the one before,
    # the last for none; the Dirichlet shell and the ghost layers follow
    nx, ny, nz, seed = 45, 21, 33, 9
    rng = np.random.default_rng(3)
    with od.Jacobi3D(nx, ny, nz, split=(3, 2, 2), seed=seed, path=path) as s:
        for scale in (1.0, 3e4, 1e200, 1.0, 1e280):
            u = rng.random(nx * ny * nz) * scale
            s.write(u)
            s.step(3)
            assert same(s.read(), solve_from(nx, ny, nz, seed, u, 3)), scale


@pytest.mark.parametrize("path", ["persistent", "per_chare", "fused_graph"])
def test_faces_fed_from_outside(od, path):
    # an imported face may hold anything: the context leaves its words
    nx, ny, nz, seed, iters = 28, 22, 19, 4, 5
    rng = np.random.default_rng(8)
    P = oracle.init_padded(nx, ny, nz, seed, 1)
    mid = oracle.sweep(P, 2)
    face = rng.random(nz * ny) * 1e290
    mid[1:-1, 1:-1, 0] = face.reshape(nz, ny)
    want = oracle.interior(oracle.sweep(mid, iters))
    with od.Jacobi3D(nx, ny, nz, split=(2, 2, 2), seed=seed, path=path) as s:
        s.step(2)
        s.face_copy(0, 1, face)  # the ghost layer of the parity that the next step reads
        s.step(1)
        s.face_copy(0, 1, face)  # and of the other one
        s.step(iters - 1)
        assert same(s.read(), want)
        out = np.empty(nz * ny)
        s.face_copy(1, 0, out)
        assert same(out, want.reshape(nz, ny, nx)[:, :, nx - 1].ravel())


@pytest.mark.parametrize("kw", [
    dict(cuts=([0, 4, 260], [0, 128], [0, 3])),                       # a tile that reads more than 19 others
    dict(cuts=([0, 1, 2, 260], [0, 1, 128], [0, 1, 3]), tile_z=1),     # single cells, rows and planes
    dict(split=(2, 2, 1), stages=3, tile_z=2), dict(split=(2, 2, 1), stages=8, tile_z=1),
    dict(split=(3, 2, 3), threads=512, cells_per_thread=1), dict(split=(1, 4, 1), threads=256, cells_per_thread=8),
])
@pytest.mark.parametrize("path", ["persistent", "fused"])
def test_tile_shapes(od, path, kw):
    want = oracle.solve(260, 128, 3, 6, 1, 7)
    with od.Jacobi3D(260, 128, 3, seed=6, path=path, **kw) as s:
        s.step(3)
        s.step(4)
        assert same(s.read(), want)


# a fused step draws tickets for the tiles past its resident CTAs (152 SMs x 6 at
# 128 x 4) and leaves the counter at zero for the next launch of any path
@pytest.mark.parametrize("tiles", [911, 912, 913, 1823, 1825, 4001])
def test_fused_tickets(od, tiles):
    want = oracle.solve(5, 2, tiles, 3, 1, 9)
    with od.Jacobi3D(5, 2, tiles, split=(1, 1, 1), seed=3, path="fused", tile_z=1, threads=128, cells_per_thread=4) as s:
        for path, n in (("fused", 3), ("persistent", 2), ("fused_graph", 1), ("fused", 2), ("persistent", 1)):
            s.set_path(path)
            s.step(n)
        assert same(s.read(), want)


@pytest.mark.parametrize("kind", ["edges", "tiny", "huge", "infinite"])
@pytest.mark.parametrize("path", ["persistent", "fused", "per_chare"])
def test_2d_fields_outside_the_window(od, path, kind):
    nx, ny, seed, iters = 143, 61, 5, 7
    u = field(kind, nx * ny, np.random.default_rng(len(kind)))
    want = solve_from(nx, ny, 0, seed, u, iters)
    with od.Jacobi2D(nx, ny, split=(3, 2), seed=seed, path=path) as s:
        s.write(u)
        s.step(iters)
        assert same(s.read(), want)


# below a million cells the entry sweeps doubles, above words; rows and planes
# that do not divide a block, one plane, one row and columns of one cell
@pytest.mark.parametrize("dims", [(7, 300, 5), (131, 127, 65), (1100, 1000, 1), (3, 1, 400000), (1, 5003, 211)])
@pytest.mark.parametrize("kind", ["uniform", "edges", "tiny", "huge"])
def test_allocation_free_entry(od, dims, kind):
    import torch
    nx, ny, nz = dims
    rng = np.random.default_rng(nx)
    P = field(kind, (nx + 2) * (ny + 2) * (nz + 2), rng).reshape(nz + 2, ny + 2, nx + 2)
    for iters in (3, 7, 8):
        want = oracle.sweep(P.copy(), iters)
        u = torch.from_numpy(P.ravel().copy()).to("cuda:0")
        out = torch.full_like(u, -1.0)
        od.jacobi_noalloc(u, out, nx, ny, nz, iters)
        torch.cuda.synchronize()
        got = out.cpu().numpy().reshape(P.shape)
        assert same(got[1:-1, 1:-1, 1:-1], want[1:-1, 1:-1, 1:-1]), iters
        shell = np.ones(P.shape, dtype=bool)
        shell[1:-1, 1:-1, 1:-1] = False
        assert same(got[shell], P[shell])  # carried over unchanged


# rows of one cell in a ring too deep for the wider tiles
@pytest.mark.parametrize("path", ["persistent", "fused", "per_chare"])
@pytest.mark.parametrize("stages", [7, 8])
def test_deep_rings_of_narrow_rows(od, path, stages):
    want = oracle.solve(1, 2048, 512, 2, 1, 3)
    with od.Jacobi3D(1, 2048, 512, split=(1, 1, 1), seed=2, path=path, stages=stages) as s:
        s.step(3)
        assert same(s.read(), want)


# faces fed before every step, whose values outgrow the window that the field's
# words have, lie far below it, or ask for plain doubles: the whole field
# follows, its other faces' shell included
@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("scales", [(1.0, 0.5, 1.0), (1.0, 3e4, 1.0, 1e200, 1e-3), (1e-9, 2.0, 1e290, 1.0)])
def test_faces_that_change_the_format(od, path, scales):
    nx, ny, nz, seed = 36, 22, 29, 4
    rng = np.random.default_rng(8)
    P = oracle.init_padded(nx, ny, nz, seed, 1)
    shell = [P[1:-1, 1:-1, 0], P[1:-1, 1:-1, -1], P[1:-1, 0, 1:-1], P[1:-1, -1, 1:-1], P[0, 1:-1, 1:-1],
             P[-1, 1:-1, 1:-1]]
    ghosts = [[a.copy() for a in shell], [a.copy() for a in shell]]  # of even and of odd steps' fields
    with od.Jacobi3D(nx, ny, nz, split=(2, 2, 2), seed=seed, path=path) as s:
        for t, scale in enumerate(scales * 2):
            f = (5 * t) % 6
            face = rng.random(shell[f].shape) * scale
            if t % 3 == 2:
                face[::4] *= -1.0
            s.face_copy(f, 1, np.ascontiguousarray(face).ravel())
            ghosts[t % 2][f][...] = face  # the field of this step's parity keeps it
            for a, g in zip(shell, ghosts[t % 2]):
                a[...] = g
            s.step(1)
            P[1:-1, 1:-1, 1:-1] = oracle.sweep(P.copy(), 1)[1:-1, 1:-1, 1:-1]
            assert same(s.read(), oracle.interior(P)), (t, scale)


def test_2d_faces_that_change_the_format(od):
    nx, ny, seed = 120, 75, 4
    rng = np.random.default_rng(8)
    P = oracle.init_padded_2d(nx, ny, seed, 1)
    with od.Jacobi2D(nx, ny, split=(2, 3), seed=seed, path="persistent") as s:
        for scale in (1.0, 5e3, 1e240, 1.0):
            face = rng.random(ny) * scale
            s.face_copy(1, 1, face)
            s.step(1)
            P[1:-1, -1] = face
            P = oracle.sweep_2d(P, 1)
            assert same(s.read(), P[1:-1, 1:-1].ravel()), scale


# planes of few cells share blocks, the last chunk of planes overlaps the one
# before; short rows and few rows are converted cell by cell; one and two planes
@pytest.mark.parametrize("dims", [(8, 8, 20011), (2, 1500, 400), (60000, 3, 7), (1, 1, 930000), (24, 22, 2503),
                                  (1100, 600, 2), (1200, 1001, 1)])
@pytest.mark.parametrize("kind", ["uniform", "tiny"])
def test_allocation_free_entry_of_narrow_and_flat_fields(od, dims, kind):
    import torch
    nx, ny, nz = dims
    rng = np.random.default_rng(nx)
    P = field(kind, (nx + 2) * (ny + 2) * (nz + 2), rng).reshape(nz + 2, ny + 2, nx + 2)
    for iters in (7, 10):
        want = oracle.sweep(P.copy(), iters)
        want[:, :, [0, -1]], want[:, [0, -1]], want[[0, -1]] = P[:, :, [0, -1]], P[:, [0, -1]], P[[0, -1]]
        u = torch.from_numpy(P.ravel().copy()).to("cuda:0")
        out = torch.full_like(u, -1.0)
        od.jacobi_noalloc(u, out, nx, ny, nz, iters)
        assert same(out.cpu().numpy().reshape(P.shape), want), iters


# fields whose updates each fit a window of their own but not the field's one: the
# sweep keeps doubles, after a call that did not and before one that does not
@pytest.mark.parametrize("dims", [(131, 127, 65), (12, 10, 10007)])
@pytest.mark.parametrize("kind", ["smooth", "hot", "signed", "nan"])
def test_allocation_free_entry_chooses_its_format(od, dims, kind):
    import torch
    nx, ny, nz = dims
    shape = (nz + 2, ny + 2, nx + 2)
    rng = np.random.default_rng(nx)

    def call(P, iters):
        want = oracle.sweep(P.copy(), iters)
        want[:, :, [0, -1]], want[:, [0, -1]], want[[0, -1]] = P[:, :, [0, -1]], P[:, [0, -1]], P[[0, -1]]
        u = torch.from_numpy(P.ravel().copy()).to("cuda:0")
        out = torch.full_like(u, -1.0)
        od.jacobi_noalloc(u, out, nx, ny, nz, iters)
        return out.cpu().numpy().reshape(shape), want

    plain = rng.random(shape)
    P = rng.random(shape)
    if kind == "smooth":
        P = np.exp2(-90.0 * np.arange(nz + 2) / nz)[:, None, None] * (0.9 + 0.1 * P)
    elif kind == "hot":
        P[nz // 2, 0, :] = 1e9
    elif kind == "signed":
        P -= 0.5
    else:
        P[nz // 2, 5, 5] = np.nan
    for field_, iters in ((plain, 8), (P, 8), (P, 9), (plain, 9)):
        got, want = call(field_, iters)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert same(np.nan_to_num(got), np.nan_to_num(want)), iters


# a context's first face import may be part of a stream capture
def test_first_face_import_under_capture(od):
    import torch
    nx, ny, nz, seed = 24, 20, 16, 3
    st = torch.cuda.Stream()
    face = torch.from_numpy(np.random.default_rng(1).random(ny * nz) * 7.0).cuda()
    P = oracle.init_padded(nx, ny, nz, seed, 1)
    with od.Jacobi3D(nx, ny, nz, split=(2, 2, 1), seed=seed, path="persistent", stream=st.cuda_stream) as s:
        s.sync()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.face_copy(0, 1, face)
        g.replay()
        torch.cuda.synchronize()
        P[1:-1, 1:-1, 0] = face.cpu().numpy().reshape(nz, ny)
        s.step(1)
        assert same(s.read(), oracle.interior(oracle.sweep(P, 1)))


# most of a signed field's cells leave the window; NaN spreads by one cell a step
@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("threads,cpt", [(128, 2), (128, 4), (256, 4), (512, 2)])
def test_signed_fields_and_nan(od, path, threads, cpt):
    nx, ny, nz, seed, iters = 62, 31, 24, 5, 5
    rng = np.random.default_rng(threads + cpt)
    u = rng.random(nx * ny * nz) - 0.5
    kw = dict(split=(2, 2, 2), seed=seed, path=path, threads=threads, cells_per_thread=cpt)
    with od.Jacobi3D(nx, ny, nz, **kw) as s:
        s.write(u)
        s.step(iters)
        assert same(s.read(), solve_from(nx, ny, nz, seed, u, iters))
        u[nx * ny * 11 + 7] = np.nan
        s.write(u)
        s.step(2)
        s.step(1)
        got, want = s.read(), solve_from(nx, ny, nz, seed, u, 3)
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(want).sum() > 20
        assert same(np.nan_to_num(got), np.nan_to_num(want))
