"""The plan that a context runs (csrc/od_plan.cpp, beside the one that od_plan
reports), built from the source on the host: what it accepts and the shared
memory that its rings leave."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_12734_gb300", "csrc")

SRC = r"""
#include <string.h>
#include "od_plan.h"
extern "C" int running_plan(const int64_t *n, const int32_t *split, int stencil, int path, int stages, int running,
                            int32_t *out) {
    od_config c;
    memset(&c, 0, sizeof c);
    c.nx = n[0]; c.ny = n[1]; c.nz = n[2];
    c.px = split[0]; c.py = split[1]; c.pz = split[2];
    c.stencil = stencil; c.path = path; c.stages = stages; c.arith = -1;
    od::Plan p;
    std::string err;
    if (od::build_plan(&c, &p, &err, true, running != 0) != OD_OK) return 1;
    const int32_t v[8] = {p.threads, p.cpt, p.stages, p.smem_bytes, (int32_t)p.tiles.size(), p.stage_doubles,
                          od::words_ctas(p.threads, p.cpt, stencil == OD_STENCIL_3D7),
                          od::words_static_smem(p.threads)};
    memcpy(out, v, sizeof v);
    return 0;
}
"""
KEYS = ("threads", "cpt", "stages", "smem", "ntiles", "slot", "ctas", "static_smem")
OPT_IN, PER_SM, RESERVED = 227 * 1024, 228 * 1024, 1024  # shared memory of a CTA, of an SM; the hardware's per CTA


@pytest.fixture(scope="module")
def running(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(SRC)
    so = str(d / "plan.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    str(d / "p.cpp"), os.path.join(CSRC, "od_plan.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def plan(dims, split, stencil=0, path=3, stages=0, run=True):
        out = (ctypes.c_int32 * 8)()
        if lib.running_plan((ctypes.c_int64 * 3)(*dims), (ctypes.c_int32 * 3)(*split), stencil, path, stages, int(run),
                            out):
            return None
        return dict(zip(KEYS, out))

    return plan


# what a plan reports as accepted, a context accepts on every path and in every
# ring depth: rows of a few cells, whose wider tiles have the most rows, and
# any others
@pytest.mark.parametrize("dims,split", [((1, 2048, 512), (1, 1, 1)), ((2, 2048, 512), (1, 1, 1)),
                                        ((3, 2048, 512), (1, 1, 1)), ((64, 700, 40), (64, 1, 1))])
def test_a_wider_shape_that_does_not_fit_is_not_run(running, dims, split):
    for path in range(5):
        for stages in (0, 3, 4, 5, 6, 7, 8):
            assert running(dims, split, path=path, stages=stages, run=False)
            p = running(dims, split, path=path, stages=stages)
            assert p is not None, (path, stages)
            # and the kernels over words fit beside their own shared memory
            assert p["smem"] + p["static_smem"] <= OPT_IN, (path, stages)


def test_what_is_reported_is_accepted(running):
    rng = random.Random(5)
    for _ in range(400):
        dims = [max(1, int(2 ** rng.uniform(0, 10))) for _ in range(3)]
        split = [rng.randint(1, max(1, min(n, 6))) for n in dims]
        stages, path = rng.choice([0, 3, 5, 7, 8]), rng.randint(0, 4)
        if running(dims, split, path=path, stages=stages, run=False):
            assert running(dims, split, path=path, stages=stages), (dims, split, stages, path)


# the ring is as deep as it can be without taking a CTA's place on the SM
@pytest.mark.parametrize("stencil", [0, 1])
def test_ring_depth_leaves_room_for_the_resident_ctas(running, stencil):
    deep = 0
    for width in range(4, 1200, 3):
        dims, split = ((width, 260, 260), (1, 1, 1)) if stencil == 0 else ((width * 4, 900, 1), (4, 3, 1))
        for path in (1, 3):
            p = running(dims, split, stencil=stencil, path=path)
            if p["stages"] > 4:
                deep += 1
                assert p["ctas"] * (p["smem"] + p["static_smem"] + RESERVED) <= PER_SM, (width, path, p)
    assert deep > 300
