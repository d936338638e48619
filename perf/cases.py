"""The solves that a user of this package runs, as timed cases.

Every case is one whole call through the public entry points on inputs a user
has in hand: a field goes in (``write``), the solver iterates it (``step``),
the result comes back (``read``) -- or the same through the server, the
allocation-free entry point, or pinned host memory.  Kinds:

* ``solve``    a field on the device through a resident context
* ``host``     a field in pinned host memory, asynchronous import and export
* ``serve``    a burst of independent jobs through ``Server``
* ``noalloc``  a padded device field through ``jacobi_noalloc``

Initial fields are the library's own seeded ones (SplitMix64 of the padded
global cell index, see ``splitmix_field``), so ``exact`` can restate them.
"""
import math

import numpy as np
import torch

from paper_2605_12734_gb300 import Jacobi2D, Jacobi3D, Server, jacobi_noalloc
from paper_2605_12734_gb300 import inputs

DEVICE = "cuda"

# The largest listed passes update 1.3e10 cells of large chares; a drawn case,
# whose chares may be small and cold, stays well below that (cell updates of
# one pass, cells of one field).
MOST_UPDATES = 5e9
MOST_CELLS_3D = 640 ** 3
MOST_CELLS_2D = 16384 ** 2


def listed():
    uneven = inputs.uneven_768()
    return [
        # the smallest call there is: the 2D smoke solve; its time is latency
        {"name": "small2d-96x64", "kind": "solve", "stencil": "2d5", "nx": 96, "ny": 64, "nz": 1, "px": 2, "py": 2,
         "pz": 1, "path": "persistent", "init_mode": 1, "iters": 7},
        # the 64^3 parity workload: cold interior, random shell, ten iterations
        {"name": "parity-64-odf8", "kind": "solve", "stencil": "3d7", "nx": 64, "ny": 64, "nz": 64, "px": 2, "py": 2,
         "pz": 2, "path": "fused", "init_mode": 0, "iters": 10},
        # one ordinary serving-sized solve alone: edge and blocks that do not divide
        {"name": "job-203-odf27", "kind": "solve", "stencil": "3d7", "nx": 203, "ny": 203, "nz": 203, "px": 3, "py": 3,
         "pz": 3, "path": "persistent", "init_mode": 1, "iters": 100},
        # the headline: 512^3 in 4096 chares of 32^3, 100 iterations
        {"name": "cube-512-odf4096", "kind": "solve", "stencil": "3d7", "nx": 512, "ny": 512, "nz": 512, "px": 16,
         "py": 16, "pz": 16, "path": "persistent", "init_mode": 1, "iters": 100},
        # the undecomposed end of the overdecomposition sweep, on the default path
        {"name": "cube-512-odf1", "kind": "solve", "stencil": "3d7", "nx": 512, "ny": 512, "nz": 512, "px": 1, "py": 1,
         "pz": 1, "path": "fused", "init_mode": 1, "iters": 20},
        # the paper's runtime flow (compute, pack, copies, unpack per chare) replayed as graphs
        {"name": "cube-512-odf64-graph", "kind": "solve", "stencil": "3d7", "nx": 512, "ny": 512, "nz": 512, "px": 4,
         "py": 4, "pz": 4, "path": "graph", "init_mode": 1, "iters": 20},
        # 300 uneven chares, as after refinement: ragged rows, slabs and chunks
        {"name": "uneven-768-300", "kind": "solve", "stencil": "3d7", "nx": uneven.nx, "ny": uneven.ny,
         "nz": uneven.nz, "cuts_seed": 25, "path": "persistent", "init_mode": 1, "iters": 50},
        # the largest resident 3D workload of the benchmark
        {"name": "cube-1024-odf4096", "kind": "solve", "stencil": "3d7", "nx": 1024, "ny": 1024, "nz": 1024, "px": 16,
         "py": 16, "pz": 16, "path": "persistent", "init_mode": 1, "iters": 12},
        # the paper's Jacobi2D base domain per GPU, overdecomposed
        {"name": "jacobi2d-32768-odf4096", "kind": "solve", "stencil": "2d5", "nx": 32768, "ny": 32768, "nz": 1,
         "px": 64, "py": 64, "pz": 1, "path": "persistent", "init_mode": 1, "iters": 16},
        # a job whose field comes from and returns to pinned host memory
        {"name": "host-256-odf64", "kind": "host", "stencil": "3d7", "nx": 256, "ny": 256, "nz": 256, "px": 4, "py": 4,
         "pz": 4, "path": "persistent", "init_mode": 1, "iters": 100},
        # a burst of requests of the serving stream's shapes
        {"name": "serve-12-jobs", "kind": "serve", "jobs": 12, "stream_seed": 6, "edge_lo": 64, "edge_hi": 256,
         "iters_lo": 10, "iters_hi": 100},
        # the largest common cube of the allocation-free entry point
        {"name": "noalloc-198", "kind": "noalloc", "nx": 198, "ny": 198, "nz": 198, "iters": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["solve3", "solve2", "host", "serve", "noalloc"], [5, 3, 1, 1, 1])[0]
    if kind == "serve":
        return {"kind": "serve", "jobs": rng.randint(2, 12), "stream_seed": rng.randint(1, 1 << 30), "edge_lo": 64,
                "edge_hi": rng.randint(96, 256), "iters_lo": 10, "iters_hi": rng.randint(20, 100)}
    if kind == "noalloc":
        nx, ny, nz = (_log_int(rng, 8, 198) for _ in range(3))
        return {"kind": "noalloc", "nx": nx, "ny": ny, "nz": nz, "iters": rng.randint(1, 40)}
    if kind == "solve2":
        nx, ny = _log_int(rng, 64, 24000), _log_int(rng, 64, 24000)
        while nx * ny > MOST_CELLS_2D:
            nx, ny = max(64, nx // 2), max(64, ny // 2)
        px, py = (min(n // 16, _log_int(rng, 1, max(1, n // 64))) for n in (nx, ny))
        most = max(1, min(200, int(MOST_UPDATES / (nx * ny))))
        return {"kind": "solve", "stencil": "2d5", "nx": nx, "ny": ny, "nz": 1, "px": max(1, px), "py": max(1, py),
                "pz": 1, "path": rng.choice(["persistent", "persistent", "fused", "fused_graph"]),
                "init_mode": rng.choice([1, 1, 1, 0]), "iters": _log_int(rng, 1, most)}
    top = 256 if kind == "host" else 900
    dims = [_log_int(rng, 32, top) for _ in range(3)]
    while dims[0] * dims[1] * dims[2] > MOST_CELLS_3D:
        dims = [max(32, int(d * 0.8)) for d in dims]
    most = max(1, min(200, int(MOST_UPDATES / (dims[0] * dims[1] * dims[2]))))
    split = [min(n // 12, _log_int(rng, 1, max(1, n // 24))) for n in dims]
    path = rng.choice(["persistent", "persistent", "persistent", "fused", "fused_graph", "graph"])
    if path == "graph":  # the per-chare flow is for few chares
        split = [min(p, 4) for p in split]
        most = min(most, 40)
    return {"kind": "host" if kind == "host" else "solve", "stencil": "3d7", "nx": dims[0], "ny": dims[1],
            "nz": dims[2], "px": split[0], "py": split[1], "pz": split[2],
            "path": "persistent" if kind == "host" else path, "init_mode": rng.choice([1, 1, 1, 0]),
            "iters": _log_int(rng, 1, most)}


def _jobs(case, seed):
    stream = inputs.serving_stream(case["jobs"], 1e6, seed=case["stream_seed"], edge_lo=case["edge_lo"],
                                   edge_hi=case["edge_hi"], iters_lo=case["iters_lo"], iters_hi=case["iters_hi"])
    return [(j.edge, j.p, j.iters, (j.seed + seed) & (2 ** 62 - 1)) for j in stream]


def _padded_noalloc(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    return torch.rand((case["nz"] + 2) * (case["ny"] + 2) * (case["nx"] + 2), generator=gen, dtype=torch.float64,
                      device=DEVICE)


def prepare(case, seed):
    if case["kind"] == "noalloc":
        field = _padded_noalloc(case, seed)
        return {"case": case, "in": field, "out": torch.empty_like(field)}
    if case["kind"] == "serve":
        jobs = _jobs(case, seed)
        need = sum(20 * (e + 2 * p) ** 3 + 200 * e * e * p + (8 << 20) for e, p, _, _ in jobs)
        outs = [torch.empty(e ** 3, dtype=torch.float64, device=DEVICE) for e, _, _, _ in jobs]
        return {"case": case, "server": Server(need), "jobs": jobs, "out": outs}
    kw = {"path": case["path"], "seed": seed, "init_mode": case["init_mode"]}
    if "cuts_seed" in case:
        kw["cuts"] = inputs.uneven_768().cuts
    else:
        kw["split"] = (case["px"], case["py"], case["pz"])
    if case["stencil"] == "2d5":
        kw["split"] = kw["split"][:2]
        ctx = Jacobi2D(case["nx"], case["ny"], **kw)
    else:
        ctx = Jacobi3D(case["nx"], case["ny"], case["nz"], **kw)
    cells = case["nx"] * case["ny"] * case["nz"]
    field = torch.empty(cells, dtype=torch.float64, device=DEVICE)
    ctx.read(field)
    if case["kind"] == "host":
        pinned = torch.empty(cells, dtype=torch.float64, pin_memory=True)
        pinned.copy_(field)
        return {"case": case, "ctx": ctx, "in": pinned, "out": torch.empty(cells, dtype=torch.float64, pin_memory=True)}
    return {"case": case, "ctx": ctx, "in": field, "out": torch.empty_like(field)}


def run(state):
    case = state["case"]
    if case["kind"] == "noalloc":
        stream = torch.cuda.current_stream().cuda_stream
        jacobi_noalloc(state["in"], state["out"], case["nx"], case["ny"], case["nz"], case["iters"], stream=stream)
        return state["out"]
    if case["kind"] == "serve":
        server = state["server"]
        ids = [server.submit(e, e, e, iters, split=(p, p, p), seed=s) for e, p, iters, s in state["jobs"]]
        for job, out in zip(ids, state["out"]):
            server.wait(job)
            server.fetch(job, out)
            server.release(job)
        return state["out"]
    ctx = state["ctx"]
    if case["kind"] == "host":
        ctx.write_async(state["in"])
        ctx.step(case["iters"])
        ctx.read_async(state["out"])
        ctx.sync()
        return state["out"]
    ctx.write(state["in"])
    ctx.step(case["iters"])
    return ctx.read(state["out"])


def work(case):
    """The field in once and out once, and per iteration one read and one write
    of every cell: an iteration's field is the next one's input.  Adds and
    divisions count one operation each."""
    if case["kind"] == "serve":
        jobs = _jobs(case, 0)
        return {"bytes": sum(8 * e ** 3 + 16 * e ** 3 * iters for e, _, iters, _ in jobs),
                "flops": sum(6 * e ** 3 * iters for e, _, iters, _ in jobs)}
    cells = case["nx"] * case["ny"] * case["nz"]
    per_cell = 4 if case.get("stencil") == "2d5" else 6
    return {"bytes": 16 * cells * (case["iters"] + 1), "flops": per_cell * cells * case["iters"]}


# ---------------------------------------------------------------- exact values


def _srl(z, n):
    """Logical right shift of an int64 tensor."""
    return (z >> n) & ((1 << (64 - n)) - 1)


def _wrap(v):
    """An unsigned 64-bit constant as the int64 of the same bits."""
    v &= 2 ** 64 - 1
    return v - 2 ** 64 if v >= 2 ** 63 else v


def splitmix_field(start, count, seed):
    """U[0,1) of padded cells start .. start+count-1: SplitMix64 output
    (cell + 1) of the seed, its top 53 bits scaled by 2^-53."""
    z = torch.arange(start + 1, start + 1 + count, dtype=torch.int64, device=DEVICE)
    z = z * _wrap(0x9E3779B97F4A7C15) + _wrap(seed)
    z = (z ^ _srl(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ _srl(z, 27)) * _wrap(0x94D049BB133111EB)
    z = z ^ _srl(z, 31)
    return _srl(z, 11).to(torch.float64) * 2.0 ** -53


def _initial(shape, seed, init_mode):
    """The padded initial field (slowest axis first)."""
    n = int(np.prod(shape))
    field = torch.empty(n, dtype=torch.float64, device=DEVICE)
    step = 1 << 26
    for at in range(0, n, step):
        field[at:at + step] = splitmix_field(at, min(step, n - at), seed)
    field = field.view(shape)
    if init_mode == 0:
        field[tuple(slice(1, -1) for _ in shape)] = 0.0
    return field


def _sweep(field, iters):
    """`iters` Jacobi sweeps of a padded field in binary64: neighbours added
    along x, then y, then z, low side first, and one division."""
    nd = field.dim()
    inner = [slice(1, -1)] * nd
    # a one-element tensor: a Python scalar would multiply by its reciprocal
    div = torch.full((1,), 2.0 * nd, dtype=torch.float64, device=field.device)
    a, b = field, field.clone()
    for _ in range(iters):
        total = None
        for axis in range(nd - 1, -1, -1):
            for side in (slice(0, -2), slice(2, None)):
                at = list(inner)
                at[axis] = side
                total = a[tuple(at)].clone() if total is None else total.add_(a[tuple(at)])
        torch.div(total, div, out=total)
        b[tuple(inner)] = total
        a, b = b, a
    return a


def _interior(field):
    return field[tuple(slice(1, -1) for _ in range(field.dim()))].reshape(-1)


def exact(case, seed):
    if case["kind"] == "noalloc":
        shape = (case["nz"] + 2, case["ny"] + 2, case["nx"] + 2)
        return _sweep(_padded_noalloc(case, seed).view(shape), case["iters"]).reshape(-1)
    if case["kind"] == "serve":
        return [_interior(_sweep(_initial((e + 2, e + 2, e + 2), s, 1), iters)) for e, _, iters, s in _jobs(case, seed)]
    if case["stencil"] == "2d5":
        shape = (case["ny"] + 2, case["nx"] + 2)
    else:
        shape = (case["nz"] + 2, case["ny"] + 2, case["nx"] + 2)
    out = _interior(_sweep(_initial(shape, seed, case["init_mode"]), case["iters"]))
    return out.cpu() if case["kind"] == "host" else out
