"""What a user of this library has it do, as measurable cases.

Every case goes through the public binding (``lbibm.Simulation``,
``lbibm.bead_relax``, the context-free ``ibm_area_volume_noalloc``) with its
default settings; sizes come from the scenes of ``scene.py``, the benchmark's
workloads and the tests.

Kinds:

* ``cycle``    one channel with bead-chain posts and cells: a few immersed-boundary
               cycles, then the node positions of every cell (asynchronous
               readback into a page-locked buffer) and the fields, as a
               trajectory recording run does between two records.
* ``batch``    the batched gap sweep: channels of uneven size in one context.
* ``gap``      the gap-threshold experiment: one cell in front of a slit per
               channel, collisions on, diagnostics and positions per channel.
* ``adjoint``  objective and gradient of the differentiable variant.
* ``beads``    overdamped assembly of magnetic beads.
* ``area``     per-cell area and volume from caller-owned device buffers.

``exact`` repeats a case in 64 bits with plain torch.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1110_0995_gb300 import lbibm, scene

WARM = 24            # cycles a state has run before it is handed out (flow and cell forces developed)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: volume and area of a filter's cells inside someone else's loop
        {"name": "area_62_cells", "kind": "area", "n_rbc": 60, "n_ctc": 2},
        # one red cell in the plain channel (the parity workload): launch latency
        {"name": "channel_32x16x64_f32", "kind": "cycle", "storage": "f32", "nx": 32, "ny": 16, "nz": 64, "cols": 0,
         "rows": 0, "n_rbc": 1, "n_ctc": 0, "force": 1e-5, "option": "none", "steps": 10},
        # bit-reproducible run of the small filter (regression runs use it)
        {"name": "small_filter_reproducible", "kind": "cycle", "storage": "f32", "nx": 96, "ny": 48, "nz": 32,
         "cols": 2, "rows": 2, "n_rbc": 4, "n_ctc": 1, "force": 2e-5, "option": "deterministic", "steps": 20},
        # odd extents: rows that break inside warps, a padded tail
        {"name": "ragged_181x75x53_f32", "kind": "cycle", "storage": "f32", "nx": 181, "ny": 75, "nz": 53, "cols": 3,
         "rows": 2, "n_rbc": 24, "n_ctc": 1, "force": 2e-5, "option": "none", "steps": 15},
        # the filter of the benchmark line, positions recorded every 10 cycles
        {"name": "filter_256x128x64_f32", "kind": "cycle", "storage": "f32", "nx": 256, "ny": 128, "nz": 64, "cols": 4,
         "rows": 3, "n_rbc": 60, "n_ctc": 2, "force": 2e-5, "option": "none", "steps": 10},
        # the same filter with half the population bytes
        {"name": "filter_256x128x64_bf16", "kind": "cycle", "storage": "bf16", "nx": 256, "ny": 128, "nz": 64,
         "cols": 4, "rows": 3, "n_rbc": 60, "n_ctc": 2, "force": 2e-5, "option": "none", "steps": 10},
        # the largest single-GPU workload, full and 16-bit storage
        {"name": "filter_512x256x128_f32", "kind": "cycle", "storage": "f32", "nx": 512, "ny": 256, "nz": 128,
         "cols": 8, "rows": 4, "n_rbc": 400, "n_ctc": 4, "force": 2e-6, "option": "none", "steps": 10},
        {"name": "filter_512x256x128_f16", "kind": "cycle", "storage": "f16", "nx": 512, "ny": 256, "nz": 128,
         "cols": 8, "rows": 4, "n_rbc": 400, "n_ctc": 4, "force": 2e-6, "option": "none", "steps": 10},
        # the gap sweep: 24 channels of uneven size in one context
        {"name": "sweep_24_channels", "kind": "batch", "storage": "f32", "channels": 24, "steps": 10},
        # the gap-threshold experiment: 16 slits, collisions, a look at every channel
        {"name": "gap_16_slits", "kind": "gap", "gaps": 8, "dims": "96x40x32", "force": 1e-5, "steps": 25},
        # gradient of the filter objective on the differentiable channel
        {"name": "adjoint_128x64x64", "kind": "adjoint", "nx": 128, "ny": 64, "nz": 64, "rows": 2, "post_beads": 6,
         "n_rbc": 8, "n_ctc": 1, "force": 1e-5, "steps": 100, "every": 50},
        # assembly of a few thousand magnetic beads
        {"name": "beads_4096", "kind": "beads", "n": 4096, "periodic": 1, "steps": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_cycle(rng):
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    option = rng.choice(["none", "none", "none", "collisions", "mass", "deterministic"])
    nx, ny, nz = _log_int(rng, 24, 480), _log_int(rng, 16, 240), _log_int(rng, 16, 120)
    if rng.random() < 0.5:                     # half of the lattices have rows that fill whole vectors
        nx = max(16, nx // 16 * 16)
    posts = rng.random() < 0.75
    cells = nx * ny * nz // 40000              # about the filter's cell density
    return {"kind": "cycle", "storage": storage, "nx": nx, "ny": ny, "nz": nz, "cols": max(1, nx // 64) if posts else 0,
            "rows": max(1, ny // 50) if posts else 0, "n_rbc": max(1, int(cells * rng.uniform(0.3, 1.2))),
            "n_ctc": rng.choice([0, 1, 2]), "force": rng.choice([2e-6, 1e-5, 2e-5]) if ny * nz < 9000 else 2e-6,
            "option": option, "steps": rng.randint(5, 24) if nx * ny * nz < 4e6 else rng.randint(3, 10)}


def draw(rng):
    kind = rng.choice(["cycle"] * 6 + ["batch", "gap", "adjoint", "beads", "area"])
    if kind == "cycle":
        return _draw_cycle(rng)
    if kind == "batch":
        return {"kind": "batch", "storage": rng.choice(["f32", "f32", "f16"]), "channels": rng.randint(2, 24),
                "steps": rng.randint(4, 10)}
    if kind == "gap":
        dims = "%dx%dx%d" % (rng.randint(84, 128), rng.randint(36, 52), rng.randint(28, 40))
        return {"kind": "gap", "gaps": rng.randint(1, 8), "dims": dims, "force": rng.choice([5e-6, 1e-5, 2e-5]),
                "steps": rng.randint(10, 40)}
    if kind == "adjoint":
        # (enough cycles for the posts to be felt by the cells: sound travels 0.58 nodes a cycle)
        nx, ny, nz = rng.randint(64, 104), rng.randint(40, 64), rng.randint(32, 64)
        return {"kind": "adjoint", "nx": nx, "ny": ny, "nz": nz, "rows": rng.randint(1, 2),
                "post_beads": rng.randint(2, 6), "n_rbc": rng.randint(1, 8), "n_ctc": rng.randint(0, 1), "force": 1e-5,
                "steps": rng.randint(70, 100), "every": rng.randint(10, 50)}
    if kind == "beads":
        return {"kind": "beads", "n": _log_int(rng, 64, 16384), "periodic": rng.randint(0, 1),
                "steps": rng.randint(1, 30)}
    return {"kind": "area", "n_rbc": _log_int(rng, 1, 400), "n_ctc": rng.randint(0, 6)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _rotations(rng, n):
    q = rng.standard_normal((n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], axis=1).reshape(n, 3, 3)


def _sites(rng, dims, radius, posts, taken, x_max):
    """Centres for cells of one radius on a shifted lattice, clear of the walls
    in y and z, of the posts (vertical chains) and of placed cells."""
    pitch = 2 * radius + 1.2
    lo = np.array([0.0, radius + 1.0, radius + 1.0])
    hi = np.array([x_max, dims[1] - radius - 2.0, dims[2] - radius - 2.0])
    if x_max >= dims[0]:
        hi[0] = dims[0] - pitch                # periodic x: the last site keeps its distance to the first one's image
    axes = []
    for a in range(3):
        room = max(hi[a] - lo[a], 0.0)
        n = int(room // pitch) + 1
        axes.append(lo[a] + rng.uniform(0.0, room - (n - 1) * pitch + 1e-9) + pitch * np.arange(n))
    if hi[1] < lo[1] or hi[2] < lo[2]:
        return np.zeros((0, 3))
    c = np.stack(np.meshgrid(*axes, indexing="ij"), axis=-1).reshape(-1, 3)

    def far(d, limit, axis2):
        d[..., 0] -= dims[0] * np.round(d[..., 0] / dims[0])
        return (np.sqrt((d[..., :axis2] ** 2).sum(-1)) > limit).all(1)

    if len(posts):
        c = c[far(c[:, None, :2] - posts[None, :, :2], radius + scene.BEAD_RADIUS + 1.5, 2)]
    for centre, r in taken:
        c = c[far(c[:, None] - centre[None, None], radius + r + 1.0, 3)]
    return c


def _place(rng, dims, spheres, n_rbc, n_ctc, x_max=None):
    """Cells of both kinds, tumor cells first, randomly turned; as many as fit
    (the sites come from the extents, so their number is the same for every
    seed, which chooses among them)."""
    posts = np.unique(np.asarray(spheres, np.float64)[:, :2], axis=0) if len(spheres) else np.zeros((0, 2))
    x_max = float(dims[0]) if x_max is None else x_max
    fixed = np.random.default_rng(list(dims))
    meshes, taken = [], []
    for kind, want, radius in (("ctc", n_ctc, scene.CTC_RADIUS), ("rbc", n_rbc, scene.RBC_RADIUS)):
        v, t = scene.cell_template(kind)
        c = _sites(fixed, dims, radius, posts, taken, x_max)
        c = c[(fixed if kind == "ctc" else rng).permutation(len(c))[:want]]
        taken += [(p, radius) for p in c]
        for centre, rot in zip(c + rng.uniform(-0.25, 0.25, c.shape), _rotations(rng, len(c))):
            meshes.append(scene.Mesh(kind, scene.quantize(v @ rot.T + centre, scene.POS_QUANTUM), t, scene.STABLE[kind]))
    return meshes


def _posts(dims, cols, rows, x_span=None, n_beads=None):
    """Post array with gaps drawn per column, the same for every seed."""
    if not cols or not rows:
        return np.zeros((0, 4), np.float32)
    fit = int((dims[2] - 0.5 - 2.5 - scene.BEAD_RADIUS) // (2 * scene.BEAD_RADIUS)) + 1
    gaps = np.random.default_rng(list(dims)).uniform(8.0, 14.0, cols)
    return scene.post_array(dims, cols, rows, max(1, min(fit, n_beads or fit)), gaps, x_span=x_span)


def _scenes(case, seed):
    """The channels of a case."""
    kind = case["kind"]
    if kind == "cycle":
        rng = _rng(seed, 1)
        dims = (case["nx"], case["ny"], case["nz"])
        spheres = _posts(dims, case["cols"], case["rows"])
        option = case["option"]
        return [scene.Scene("cycle", dims, body_force=(case["force"], 0.0, 0.0), spheres=spheres,
                            meshes=_place(rng, dims, spheres, case["n_rbc"], case["n_ctc"]),
                            repulsion=(0.01, 1.0) if option == "collisions" else None,
                            ib_dynamics=(0.05, 5.0) if option == "mass" else None)]
    if kind == "batch":
        out = []
        shape = np.random.default_rng(21)      # extents as in the gap sweep, the same for every seed
        for k in range(case["channels"]):
            rng = _rng(seed, 100 + k)
            dims = (int(shape.integers(8, 33)) * 8, int(shape.integers(4, 17)) * 8, int(shape.integers(4, 9)) * 8)
            gap, n_rbc = float(shape.uniform(6.0, 16.0)), int(shape.integers(10, 41))
            shape.integers(0, 2 ** 31)         # (scene.gap_sweep draws a seed for each channel here)
            fit = int((dims[2] - 0.5 - 2.5 - scene.BEAD_RADIUS) // (2 * scene.BEAD_RADIUS)) + 1
            rows = max(1, int((dims[1] - 1) // (2 * scene.BEAD_RADIUS + gap)))
            spheres = scene.post_array(dims, 1, rows, fit, [gap], x_span=(0.0, float(dims[0])))
            out.append(scene.Scene("sweep", dims, body_force=(1e-5, 0.0, 0.0), spheres=spheres,
                                   meshes=_place(rng, dims, spheres, n_rbc, 0)))
        return out
    if kind == "gap":
        rng = _rng(seed, 2)
        dims = tuple(int(v) for v in case["dims"].split("x"))
        out = []
        for cell in ("rbc", "ctc"):
            for k in range(case["gaps"]):
                sc = scene.gap_cell(cell, 2.0 + 2.0 * k, dims, body_force=case["force"])
                m = sc.meshes[0]
                m.rest = scene.quantize(m.rest + rng.uniform(-0.5, 0.5, 3), scene.POS_QUANTUM)
                out.append(sc)
        return out
    if kind == "adjoint":
        rng = _rng(seed, 3)
        dims = (case["nx"], case["ny"], case["nz"])
        half = dims[0] / 2.0
        spheres = _posts(dims, 1, case["rows"], x_span=(half, float(dims[0])), n_beads=case["post_beads"])
        return [scene.Scene("adjoint", dims, body_force=(case["force"], 0.0, 0.0), spheres=spheres,
                            meshes=_place(rng, dims, np.zeros((0, 4)), case["n_rbc"], case["n_ctc"], x_max=half - 12.0))]
    raise ValueError(kind)


def _deformed(scenes, seed):
    """Current positions of every cell: the rest shape stretched by a few per
    cent along a random direction, as cells in the flow are."""
    rng = _rng(seed, 4)
    out = []
    for sc in scenes:
        now = []
        for m in sc.meshes:
            d = rng.standard_normal(3)
            d /= np.linalg.norm(d)
            eps = rng.uniform(0.01, 0.04)
            c = m.rest.mean(0)
            stretch = np.eye(3) * (1.0 - 0.5 * eps) + 1.5 * eps * np.outer(d, d)
            now.append(scene.quantize((m.rest - c) @ stretch + c, scene.POS_QUANTUM))
        out.append(now)
    return out


def _bead_inputs(case, seed):
    """Beads on a loose jittered lattice, moments mostly along z (a bias field)."""
    rng = _rng(seed, 5)
    n = case["n"]
    side = math.ceil(n ** (1.0 / 3.0))
    pitch = 2.6
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n]
    x = (g + 0.5) * pitch + rng.uniform(-0.35, 0.35, (n, 3))
    m = np.array([0.0, 0.0, 1.0]) + 0.2 * rng.standard_normal((n, 3))
    return x.astype(np.float32).astype(np.float64), m.astype(np.float32).astype(np.float64), side * pitch


BEADS = {"c": 0.05, "radius": 1.0, "k": 2.0, "mobility": 0.1, "dt": 0.05}


def _area_meshes(case, seed):
    rng = _rng(seed, 6)
    xyz, tris, start, base = [], [], [0], 0
    for kind, count in (("ctc", case["n_ctc"]), ("rbc", case["n_rbc"])):
        v, t = scene.cell_template(kind)
        for rot in _rotations(rng, count):
            xyz.append(v @ rot.T * rng.uniform(0.95, 1.05, 3) + rng.uniform(8.0, 200.0, 3))
            tris.append(t + base)
            base += len(v)
            start.append(start[-1] + len(t))
    return np.concatenate(xyz), np.concatenate(tris).astype(np.int32), np.array(start, np.int32)


def _pinned(n):
    return torch.empty((max(n, 1), 3), dtype=torch.float64, pin_memory=True).numpy()[:n]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "beads":
        x, m, box = _bead_inputs(case, seed)
        return {"case": case, "x": x, "m": m, "box": box}
    if kind == "area":
        xyz, tris, start = _area_meshes(case, seed)
        dev = {"xyz": torch.from_numpy(xyz).cuda(), "tris": torch.from_numpy(tris).cuda(),
               "start": torch.from_numpy(start).cuda()}
        n = len(start) - 1
        return {"case": case, "start_host": start, "n": n, "stream": torch.cuda.current_stream().cuda_stream,
                "area": torch.zeros(n, dtype=torch.float64, device="cuda"),
                "volume": torch.zeros(n, dtype=torch.float64, device="cuda"), **dev}
    scenes = _scenes(case, seed)
    if kind == "adjoint":
        bare = [scene.Scene("adjoint", s.dims, body_force=s.body_force, meshes=s.meshes) for s in scenes]
        sim = lbibm.Simulation.from_scenes(bare)
        sim.set_brinkman(np.asarray(scenes[0].spheres, np.float64))
    else:
        sim = lbibm.Simulation.from_scenes(scenes, case.get("storage", "f32"))
        if case.get("option") == "deterministic":
            sim.set_deterministic(True)
    for ch, now in enumerate(_deformed(scenes, seed)):
        sim.select(ch)
        for k, x in enumerate(now):
            sim.set_nodes(k, x)
    sim.select(0)
    sim.step(WARM)
    state = {"case": case, "sim": sim}
    if kind == "adjoint":
        return state
    state["x"] = [_pinned(sum(m.n_nodes for m in s.meshes)) for s in scenes]
    if kind in ("cycle", "batch"):
        n = sum(s.n_nodes for s in scenes)
        state["rho"] = torch.empty(n, dtype=torch.float32, device="cuda")
        state["u"] = torch.empty(3 * n, dtype=torch.float32, device="cuda")
        state["first"] = np.concatenate([[0], np.cumsum([s.n_nodes for s in scenes])]).tolist()
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "beads":
        x = lbibm.bead_relax(state["x"], state["m"], BEADS["c"], BEADS["radius"], BEADS["k"], BEADS["mobility"],
                             BEADS["dt"], case["steps"], box=(state["box"],) * 3, periodic=(case["periodic"],) * 3)
        return x.astype(np.float32)            # the library computes bead positions in FP32
    if kind == "area":
        ptr = ctypes.c_void_p
        st = lbibm.lib().ibm_area_volume_noalloc(
            ptr(state["xyz"].data_ptr()), ptr(state["tris"].data_ptr()), ptr(state["start"].data_ptr()),
            state["start_host"].ctypes.data_as(ptr), state["n"], ptr(state["area"].data_ptr()),
            ptr(state["volume"].data_ptr()), ptr(state["stream"]))
        if st != lbibm.LB_OK:
            raise lbibm.LbError(st, "ibm_area_volume_noalloc")
        return [state["area"], state["volume"]]
    sim = state["sim"]
    if kind == "adjoint":
        r = sim.adjoint(case["steps"], case["every"])
        return [r["J"], r["beads"], r["ks"], r["kb"]]
    sim.step(case["steps"])
    if kind == "gap":
        # as the gap-threshold experiment looks at its channels between two chunks of cycles
        diag = np.zeros((len(state["x"]), 6))
        for ch, x in enumerate(state["x"]):
            sim.select(ch)
            diag[ch] = sim.diagnostics()
            sim.all_nodes_into(x)
        return [np.concatenate(state["x"]), diag]
    for ch, x in enumerate(state["x"]):
        sim.select(ch)
        sim.all_nodes_into_async(x, 0)
    rho, u = state["rho"], state["u"]
    for ch in range(len(state["x"])):
        sim.select(ch)
        at = 4 * state["first"][ch]
        sim.fields_to_device(rho.data_ptr() + at, u.data_ptr() + 3 * at)
    sim.wait_readback(0)
    return [np.concatenate(state["x"]) if len(state["x"]) > 1 else state["x"][0], rho, u]


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------

def _solid(sc):
    """Obstacle nodes (inside or on a bead) as a (nz, ny, nx) array."""
    nx, ny, nz = sc.dims
    solid = np.zeros((nz, ny, nx), bool)
    for cx, cy, cz, r in np.asarray(sc.spheres, np.float64):
        lo = [max(0, math.ceil(v - r)) for v in (cx, cy, cz)]
        hi = [min(n - 1, math.floor(v + r)) for v, n in zip((cx, cy, cz), sc.dims)]
        if any(b < a for a, b in zip(lo, hi)):
            continue
        x, y, z = (np.arange(a, b + 1) for a, b in zip(lo, hi))
        d2 = (x - cx)[None, None, :] ** 2 + (y - cy)[None, :, None] ** 2 + (z - cz)[:, None, None] ** 2
        solid[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1] |= d2 <= r * r
    return solid


def work(case):
    kind = case["kind"]
    if kind == "beads":
        pairs = float(case["n"]) * case["n"]
        return {"bytes": 72.0 * case["n"], "flops": 45.0 * pairs * case["steps"]}
    if kind == "area":
        nodes, tris = 642 * case["n_rbc"] + 2562 * case["n_ctc"], 1280 * case["n_rbc"] + 5120 * case["n_ctc"]
        return {"bytes": 24.0 * nodes + 12.0 * tris + 20.0 * (case["n_rbc"] + case["n_ctc"]), "flops": 50.0 * tris}
    scenes = _scenes(case, 0)
    pop = 2 * 19 * (4 if case.get("storage", "f32") == "f32" else 2)
    fluid = sum(s.n_nodes - int(_solid(s).sum()) for s in scenes) if kind != "adjoint" else scenes[0].n_nodes
    points = sum(s.n_ib_nodes for s in scenes)
    tris = sum(m.n_tris for s in scenes for m in s.meshes)
    # a cycle reads and writes every population once; a point's position is read and written, its element
    # data (two triangles: indices and rest area; three edges: indices, rest length and angle) read once
    cycle_bytes = float(pop) * fluid + 48.0 * points + 20.0 * tris + 32.0 * 1.5 * tris
    cycle_flops = 260.0 * fluid + 1500.0 * points
    steps = case["steps"]
    if kind == "adjoint":
        # forward cycles once with their data kept and, per cycle in reverse, the stored populations and
        # the incoming adjoint read, the outgoing adjoint written (228 bytes per node)
        return {"bytes": steps * (cycle_bytes + 228.0 * fluid + 200.0 * points),
                "flops": steps * (cycle_flops + 600.0 * fluid + 6000.0 * points)}
    # fields: the populations once more and four floats per node; diagnostics: the populations once more
    end = 24.0 * points + (0.5 * pop * fluid + 16.0 * fluid if kind != "gap" else 0.5 * pop * fluid)
    return {"bytes": steps * cycle_bytes + end, "flops": steps * cycle_flops + 60.0 * fluid}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

_E = [(0, 0, 0)] + [s for a in ((1, 0, 0), (0, 1, 0), (0, 0, 1)) for s in (a, tuple(-v for v in a))]
_E += [s for a in ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)) for s in (a, tuple(-v for v in a))]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12


def _opposite(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


def _edges_of(tris):
    """(a, b, c, d): edge a < b between the triangles (a, b, c) and (b, a, d)."""
    third = {}
    for t in tris.tolist():
        for k in range(3):
            third[t[k], t[(k + 1) % 3]] = t[(k + 2) % 3]
    return np.array([(a, b, c, third[b, a]) for (a, b), c in third.items() if a < b])


class _Exact:
    """One channel in 64 bits: BGK with Guo forcing, halfway bounce-back,
    trilinear immersed boundary, elastic cells, optional collisions, points
    with mass or Brinkman beads."""

    def __init__(self, sc, now, device, brinkman=None):
        nx, ny, nz = self.dims = sc.dims
        self.dev, self.tau, self.per = device, sc.tau, sc.periodic
        self.G = torch.tensor(sc.body_force, dtype=torch.float64, device=device).reshape(3, 1, 1, 1)
        self.w = torch.tensor(_W, dtype=torch.float64, device=device).reshape(19, 1, 1, 1)
        self.solid = torch.from_numpy(_solid(sc)).to(device)
        # links that bounce back: the pull source lies outside the domain or on an obstacle
        self.bounce = []
        for i, e in enumerate(_E):
            b = torch.roll(self.solid, (e[2], e[1], e[0]), (0, 1, 2)).clone()
            for axis, (c, n) in enumerate(zip(e, sc.dims)):
                if c and not sc.periodic[axis]:
                    b.select(2 - axis, 0 if c > 0 else n - 1).fill_(True)
            self.bounce.append(b)
        self.f = self.w.expand(19, nz, ny, nx).clone()
        self.u = torch.zeros(3, nz, ny, nx, dtype=torch.float64, device=device)
        self.rho = torch.ones(nz, ny, nx, dtype=torch.float64, device=device)
        self.brinkman = brinkman                  # alpha phi per node, or None
        self._cells(sc, now)

    def _cells(self, sc, now):
        put = lambda a, t=torch.float64: torch.as_tensor(np.asarray(a), dtype=t, device=self.dev)  # noqa: E731
        self.n_cells = len(sc.meshes)
        if not self.n_cells:
            return
        rest, tris, tcell, edges, ecell, ncell, base, cache = [], [], [], [], [], [], 0, {}
        for c, m in enumerate(sc.meshes):
            key = m.tris.tobytes()
            if key not in cache:
                cache[key] = _edges_of(m.tris)
            rest.append(m.rest)
            tris.append(m.tris + base)
            edges.append(cache[key] + base)
            tcell += [c] * m.n_tris
            ecell += [c] * len(cache[key])
            ncell += [c] * m.n_nodes
            base += m.n_nodes
        self.rest, self.x = put(np.concatenate(rest)), put(np.concatenate(now))
        self.tri, self.edge = put(np.concatenate(tris), torch.int64), put(np.concatenate(edges), torch.int64)
        self.tcell, self.ecell, self.ncell = (put(v, torch.int64) for v in (tcell, ecell, ncell))
        self.mod = put([m.moduli for m in sc.meshes])
        a, b = self.rest[self.edge[:, 0]], self.rest[self.edge[:, 1]]
        self.L0 = (b - a).norm(dim=1)
        self.th0 = self._dihedral(self.rest)[0]
        self.S0t = 0.5 * self._normal(self.rest)[0].norm(dim=1)
        self.S0, self.V0 = self._totals(self.rest)
        self.beads = put(np.asarray(sc.spheres, np.float64).reshape(-1, 4))
        self.rep = sc.repulsion
        self.mass = sc.ib_dynamics
        self.v = torch.zeros_like(self.x)

    def _normal(self, x):
        a, b, c = (x[self.tri[:, k]] for k in range(3))
        return torch.linalg.cross(b - a, c - a), b - a, c - a

    def _totals(self, x):
        n = self._normal(x)[0]
        a, b, c = (x[self.tri[:, k]] for k in range(3))
        zero = torch.zeros(self.n_cells, dtype=torch.float64, device=self.dev)
        vol = (a * torch.linalg.cross(b, c)).sum(1) / 6.0
        return zero.index_add(0, self.tcell, 0.5 * n.norm(dim=1)), zero.index_add(0, self.tcell, vol)

    def _dihedral(self, x):
        a, b, c, d = (x[self.edge[:, k]] for k in range(4))
        e, ac, ad = b - a, c - a, d - a
        n1, n2 = torch.linalg.cross(e, ac), torch.linalg.cross(ad, e)
        ln = e.norm(dim=1)
        theta = torch.atan2((torch.linalg.cross(n1, n2) * e).sum(1) / ln, (n1 * n2).sum(1))
        return theta, e, ac, ad, n1, n2, ln

    def forces(self, x, mod):
        """Membrane (and collision) forces on every point."""
        F = torch.zeros_like(x)
        ks, kb = mod[self.ecell, 0], mod[self.ecell, 1]
        theta, e, ac, ad, n1, n2, ln = self._dihedral(x)
        lam = ln / self.L0
        T = ks * (lam.sqrt() + lam ** -2.5) / (lam + lam ** -3) * (lam - 1.0)
        fs = (T / ln)[:, None] * e
        coef = (-kb * (theta - self.th0))[:, None]
        gc = -(ln / (n1 * n1).sum(1))[:, None] * n1
        gd = -(ln / (n2 * n2).sum(1))[:, None] * n2
        s, t = ((v * e).sum(1, keepdim=True) / (ln * ln)[:, None] for v in (ac, ad))
        for k, f in enumerate((fs + coef * ((s - 1.0) * gc + (t - 1.0) * gd), -fs - coef * (s * gc + t * gd), coef * gc,
                               coef * gd)):
            F = F.index_add(0, self.edge[:, k], f)
        n, e1, e2 = self._normal(x)
        St = 0.5 * n.norm(dim=1)
        S, V = self._totals(x)
        third = (e1 + e2) / 3.0
        ws = (-third, e1 - third, e2 - third)
        ww = sum((w * w).sum(1) for w in ws)
        tm = mod[self.tcell]
        rel = ((S - self.S0) / self.S0)[self.tcell], ((V - self.V0) / self.V0)[self.tcell]
        ca = ((tm[:, 2] * (St - self.S0t) / self.S0t + tm[:, 3] * rel[0]) * (-2.0 * St / ww))[:, None]
        fv = (tm[:, 4] * rel[1] / 6.0)[:, None] * n
        for k, w in enumerate(ws):
            F = F.index_add(0, self.tri[:, k], ca * w - fv)
        return F if self.rep is None else F + self._collisions(x)

    def _image(self, d):
        d = d.clone()
        for a in range(3):
            if self.per[a]:
                d[..., a] -= self.dims[a] * torch.round(d[..., a] / self.dims[a])
        return d

    def _collisions(self, x):
        k, dc = self.rep
        F = torch.zeros_like(x)
        if len(self.beads):
            for i in range(0, len(x), 8192):
                d = self._image(x[i:i + 8192, None] - self.beads[None, :, :3])
                ln = d.norm(dim=2)
                push = torch.where(ln < self.beads[None, :, 3] + dc, k * (dc - (ln - self.beads[None, :, 3])) / ln, 0.0)
                F[i:i + 8192] += (push[..., None] * d).sum(1)
        if self.n_cells > 1:
            for i in range(0, len(x), 2048):
                d = self._image(x[i:i + 2048, None] - x[None])
                ln = d.norm(dim=2)
                near = (ln < dc) & (ln > 0) & (self.ncell[i:i + 2048, None] != self.ncell[None])
                F[i:i + 2048] += (torch.where(near, k * (dc - ln) / ln, 0.0)[..., None] * d).sum(1)
        for a in range(3):
            if not self.per[a]:
                lo, hi = x[:, a] + 0.5, self.dims[a] - 0.5 - x[:, a]
                F[:, a] += k * ((dc - lo).clamp(min=0.0) - (dc - hi).clamp(min=0.0))
        return F

    def _stencil(self, x):
        """Flat node indices and weights of every point's eight corners
        (obstacles and nodes outside the domain have weight 0)."""
        nx, ny, nz = self.dims
        base = torch.floor(x.detach())
        fr = x - base
        idx, wts = [], []
        for c in range(8):
            w, ok, at = 1.0, True, []
            for a in range(3):
                bit = (c >> a) & 1
                w = w * (fr[:, a] if bit else 1.0 - fr[:, a])
                v = base[:, a].long() + bit
                if self.per[a]:
                    v = v % self.dims[a]
                else:
                    ok = ok & (v >= 0) & (v < self.dims[a])
                    v = v.clamp(0, self.dims[a] - 1)
                at.append(v)
            g = at[0] + nx * (at[1] + ny * at[2])
            ok = ok & ~self.solid.reshape(-1)[g]
            idx.append(g)
            wts.append(torch.where(ok, w, 0.0))
        return torch.stack(idx), torch.stack(wts)

    def _collide(self, f, g, out=None):
        """Post-collision populations, density and force-corrected velocity."""
        rho = f.sum(0)
        j = torch.stack([sum(f[i] * e[a] for i, e in enumerate(_E) if e[a]) for a in range(3)])
        if self.brinkman is None:
            u, gt = (j + 0.5 * g) / rho, g
        else:
            v, D = j + 0.5 * g, 1.0 + 0.5 * self.brinkman
            u, gt = v / (rho * D), g - self.brinkman * v / D
        om, fp = 1.0 / self.tau, 1.0 - 0.5 / self.tau
        uu, ug = (u * u).sum(0), (u * gt).sum(0)
        post = []
        for i, e in enumerate(_E):
            eu = sum(e[a] * u[a] for a in range(3) if e[a]) if i else 0.0
            eg = sum(e[a] * gt[a] for a in range(3) if e[a]) if i else 0.0
            p = (1.0 - om) * f[i] + _W[i] * (om * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu) +
                                             fp * (3.0 * (eg - ug) + 9.0 * eu * eg))
            if out is None:
                post.append(p)
            else:
                out[i] = p
        return (torch.stack(post) if out is None else out), rho, u

    def step(self):
        """One cycle in place (no gradients)."""
        nodes = self.solid.numel()
        g = self.G.expand(3, *self.solid.shape)
        if self.n_cells:
            idx, wts = self._stencil(self.x)
            F = self.forces(self.x, self.mod)
            J = F
            if self.mass is not None:
                m, gamma = self.mass
                a = gamma / m
                p1 = -math.expm1(-a) / a
                U = (wts[..., None] * self.u.reshape(3, nodes).T[idx]).sum(0)
                D = self.v + F / m - U
                J = gamma * p1 * D
                self.v = U + math.exp(-a) * D
                step = U + p1 * D
            spread = torch.zeros(nodes, 3, dtype=torch.float64, device=self.dev)
            spread.index_add_(0, idx.reshape(-1), (wts[..., None] * J[None]).reshape(-1, 3))
            g = g + spread.T.reshape(3, *self.solid.shape)
        post, self.rho, self.u = self._collide(self.f, g, out=torch.empty_like(self.f))
        post[:, self.solid] = self.w.reshape(19, 1)
        self.rho[self.solid] = 1.0
        self.u[:, self.solid] = 0.0
        self.mom = [sum(post[i] * e[a] for i, e in enumerate(_E) if e[a]) for a in range(3)]
        for i, e in enumerate(_E):
            self.f[i] = torch.where(self.bounce[i], post[_opposite(i)], torch.roll(post[i], (e[2], e[1], e[0]), (0, 1, 2)))
        self.f[:, self.solid] = self.w.reshape(19, 1)
        if self.n_cells:
            if self.mass is None:
                step = (wts[..., None] * self.u.reshape(3, nodes).T[idx]).sum(0)
            self.x = self.x + step

    def cycle(self, f, x, mod):
        """One differentiable cycle: the next populations and positions."""
        nodes = self.solid.numel()
        idx, wts = self._stencil(x)
        F = self.forces(x, mod)
        spread = torch.zeros(nodes, 3, dtype=torch.float64, device=self.dev)
        spread = spread.index_add(0, idx.reshape(-1), (wts[..., None] * F[None]).reshape(-1, 3))
        post, _, u = self._collide(f, self.G + spread.T.reshape(3, *self.solid.shape))
        nxt = torch.stack([torch.where(self.bounce[i], post[_opposite(i)], torch.roll(post[i], (e[2], e[1], e[0]), (0, 1, 2)))
                           for i, e in enumerate(_E)])
        return nxt, x + (wts[..., None] * u.reshape(3, nodes).T[idx]).sum(0)


def _exact_adjoint(case, seed, dev):
    from torch.utils.checkpoint import checkpoint

    sc = _scenes(case, seed)[0]
    now = _deformed([sc], seed)[0]
    beads = torch.tensor(np.asarray(sc.spheres, np.float64), device=dev)
    centres = beads[:, :3].clone().requires_grad_(True)
    z, y, x = torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device=dev) for n in sc.dims[::-1]], indexing="ij")
    grid = torch.stack([x, y, z])

    def alpha_phi(c):
        keep = torch.ones_like(grid[0])
        for k in range(len(beads)):
            d = (grid - c[k].reshape(3, 1, 1, 1)).square().sum(0).sqrt()
            keep = keep * (1.0 - 0.5 * (1.0 - torch.tanh((d - beads[k, 3]) / 0.5)))
        return 2.0 * (1.0 - keep)

    bare = scene.Scene("adjoint", sc.dims, body_force=sc.body_force, meshes=sc.meshes)
    S = _Exact(bare, now, dev, alpha_phi(centres.detach()))
    with torch.no_grad():
        for _ in range(WARM):
            S.step()
    x0 = S.x
    phi = alpha_phi(centres)
    moduli = S.mod[0, :2].clone().requires_grad_(True)

    def some(f, xs, a, m, n):
        S.brinkman = a
        mod = torch.cat([torch.cat([m, S.mod[0, 2:]])[None], S.mod[1:]])
        for _ in range(n):
            f, xs = S.cycle(f, xs, mod)
        return f, xs

    f, xs, left = S.f, S.x, case["steps"]
    while left:
        n = min(10, left)
        f, xs = checkpoint(some, f, xs, phi, moduli, n, use_reentrant=False)
        left -= n
    n0 = sc.meshes[0].n_nodes
    J = xs[:n0, 0].mean() - x0[:n0, 0].mean()
    gb, gm = torch.autograd.grad(J, [centres, moduli])
    return [J.detach().cpu().numpy(), gb.cpu().numpy(), gm[0].cpu().numpy(), gm[1].cpu().numpy()]


def _exact_beads(case, seed, dev):
    x, m, box = _bead_inputs(case, seed)
    x, m = torch.tensor(x, device=dev), torch.tensor(m, device=dev)
    for _ in range(case["steps"]):
        F = torch.zeros_like(x)
        for i in range(0, len(x), 512):
            r = x[i:i + 512, None] - x[None]
            if case["periodic"]:
                r = r - box * torch.round(r / box)
            d2 = (r * r).sum(2)
            d2[d2 == 0] = math.inf
            ma, mb = m[None], m[i:i + 512, None]
            mar, mbr, mab = (ma * r).sum(2), (mb * r).sum(2), (ma * mb).sum(2)
            d = d2.sqrt()
            f = (3.0 * BEADS["c"] * d ** -5)[..., None] * (mar[..., None] * mb + mbr[..., None] * ma +
                                                          (mab - 5.0 * mar * mbr / d2)[..., None] * r)
            f = f + (BEADS["k"] * (2.0 * BEADS["radius"] - d).clamp(min=0.0) / d)[..., None] * r
            F[i:i + 512] = f.sum(1)
        x = x + BEADS["mobility"] * BEADS["dt"] * F
        if case["periodic"]:
            x = x - box * torch.floor(x / box)
    return x.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "adjoint":
        return _exact_adjoint(case, seed, dev)
    if kind == "beads":
        return _exact_beads(case, seed, dev)
    if kind == "area":
        xyz, tris, start = _area_meshes(case, seed)
        a, b, c = (xyz[tris[:, k]] for k in range(3))
        area = 0.5 * np.linalg.norm(np.cross(b - a, c - a), axis=1)
        volume = (a * np.cross(b, c)).sum(1) / 6.0
        return [np.add.reduceat(area, start[:-1]), np.add.reduceat(volume, start[:-1])]
    scenes = _scenes(case, seed)
    xs, rhos, us, diags = [], [], [], []
    for sc, now in zip(scenes, _deformed(scenes, seed)):
        S = _Exact(sc, now, dev)
        for _ in range(WARM + case["steps"]):
            S.step()
        xs.append(S.x.cpu().numpy() if S.n_cells else np.zeros((0, 3)))
        if kind == "gap":
            fluid = ~S.solid
            diags.append([float(S.rho[fluid].sum())] + [float(m[fluid].sum()) for m in S.mom] +
                         [0.0, float((S.u * S.u).sum(0).max().sqrt())])
        else:
            rhos.append(S.rho.reshape(-1))
            us.append(S.u.reshape(-1))
    if kind == "gap":
        return [np.concatenate(xs), np.array(diags)]
    return [np.concatenate(xs), torch.cat(rhos), torch.cat(us)]
