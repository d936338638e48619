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


@pytest.mark.parametrize("two", [False, True])
def test_arena_holds_the_running_tiles(od, two):
    rng = random.Random(17)
    finer = 0
    for _ in range(150):
        d, kw = grid(rng, two)
        kw["tile_y"] = rng.choice([0, 0, 3, 7])
        info = od.plan(*d, **kw)
        kw.update(threads=info["threads"], cells_per_thread=info["cells_per_thread"])
        plans = {z: od.plan(*d, tile_z=z, **kw) for z in (2, 4, 8, 16, 32, 64)}
        tz = 64 if two else 32
        enough = 900 if info["threads"] >= 256 else 1800
        while tz > 4 and plans[tz]["ntiles"] < enough:
            tz //= 2
        if tz == 4 and plans[4]["ntiles"] < 800:
            tz = 2
        finer += tz < 32
        assert info["ntiles"] == plans[32]["ntiles"]
        assert info["arena_bytes"] == max(plans[32]["arena_bytes"], plans[tz]["arena_bytes"])
    assert finer > 100


def test_arena_of_a_wider_running_shape(od):
    # 64-cell rows: reported 128 x 4, run 256 x 4, whose tables are smaller
    kw = dict(split=(4, 4, 4))
    info = od.plan(256, 256, 256, **kw)
    assert (info["threads"], info["cells_per_thread"]) == (128, 4)
    wide = od.plan(256, 256, 256, threads=256, cells_per_thread=4, tile_z=16, **kw)
    assert info["arena_bytes"] >= wide["arena_bytes"]
    assert info["arena_bytes"] == max(wide["arena_bytes"], od.plan(256, 256, 256, threads=128, cells_per_thread=4,
                                                                   tile_z=32, **kw)["arena_bytes"])
