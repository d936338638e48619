"""The arena that od_plan asks for holds the tables of the tiles a context
runs with, whose planes per tile follow the grid's size: its size is that of
the larger of the two tilings, each planned explicitly."""
import random

import pytest

from paper_2605_12734_gb300 import build as od_build


@pytest.fixture(scope="module")
def od():
    od_build.build()
    import paper_2605_12734_gb300 as pkg
    return pkg


def grid(rng, two):
    def cuts(n, p):
        return [0] + sorted(rng.sample(range(1, n), p - 1)) + [n]
    d = [rng.randint(4, 160) for _ in range(3)]
    if two:
        d = [d[0] * rng.choice([1, 20]), d[1], 1]
        return d, dict(stencil="2d5", cuts=(cuts(d[0], rng.randint(1, 4)), cuts(d[1], rng.randint(1, 4))))
    return d, dict(cuts=tuple(cuts(n, rng.randint(1, min(4, n))) for n in d))


def running_shape(d, kw, shape, fused):
    """The CTA shape a context runs where a plan reports ``shape``: twice the
    cells while the rows of the blocks fill them as well, and for fused steps
    three waves of tiles where that is 256 x 4."""
    if "stencil" in kw or kw["tile_y"] or shape not in ((128, 2), (128, 4)) or d[0] * d[1] * d[2] < 1 << 19:
        return shape

    def lengths(cuts):
        return [b - a for a, b in zip(cuts, cuts[1:])]

    def slabs(cap):
        return sum(-(-h // min(h, cap // w)) for w in lengths(kw["cuts"][0]) for h in lengths(kw["cuts"][1]))

    if shape == (128, 2) and 2 * slabs(512) <= slabs(256):
        shape = (128, 4)
    if shape == (128, 4) and 2 * slabs(1024) <= slabs(512) and d[0] * d[1] * 8 >= slabs(1024) * 1024 * 5:
        if not fused or slabs(1024) * sum(-(-z // 32) for z in lengths(kw["cuts"][2])) >= 1368:
            shape = (256, 4)
    return shape


@pytest.mark.parametrize("two", [False, True])
def test_arena_holds_the_running_tiles(od, two):
    rng = random.Random(17)
    finer = wider = 0
    for _ in range(150):
        d, kw = grid(rng, two)
        kw["tile_y"] = rng.choice([0, 0, 3, 7])
        info = od.plan(*d, **kw)
        shape = (info["threads"], info["cells_per_thread"])
        here = od.plan(*d, tile_z=32, threads=shape[0], cells_per_thread=shape[1], **kw)
        bytes_ = [here["arena_bytes"]]
        for fused in (False, True):
            run = running_shape(d, kw, shape, fused)
            wider += run != shape
            plans = {z: od.plan(*d, tile_z=z, threads=run[0], cells_per_thread=run[1], **kw)
                     for z in (2, 4, 8, 16, 32, 64)}
            tz = 64 if two else 32
            enough = 900 if run[0] >= 256 else 1800
            while tz > 4 and plans[tz]["ntiles"] < enough:
                tz //= 2
            if tz == 4 and plans[4]["ntiles"] < 800:
                tz = 2
            finer += tz < 32
            bytes_.append(plans[tz]["arena_bytes"])
        assert info["ntiles"] == here["ntiles"]
        assert info["arena_bytes"] == max(bytes_)
    assert wider > 10 or two
    assert finer > 100


def test_arena_of_a_wider_running_shape(od):
    # 64-cell rows: reported 128 x 4; run 256 x 4, or for fused steps 128 x 4,
    # with 16 planes per tile either way
    kw = dict(split=(4, 4, 4))
    info = od.plan(256, 256, 256, **kw)
    assert (info["threads"], info["cells_per_thread"]) == (128, 4)
    runs = [od.plan(256, 256, 256, threads=t, cells_per_thread=4, tile_z=16, **kw) for t in (256, 128)]
    assert info["arena_bytes"] == max(r["arena_bytes"] for r in runs)
    for path in ("persistent", "fused_graph", "graph"):
        assert od.plan(256, 256, 256, path=path, **kw)["arena_bytes"] == info["arena_bytes"]
