"""The work that users of this framework have it do, as cases that can be timed.

A case is one call pattern (``kind``) on one grid and one kind of field:

* ``compute``   a plan that is kept and run on a field in device memory (a time step, a scan), then
                every output of the pass, the plan's own memory copied where the program keeps it;
* ``fresh``     ``msc.compute(field)`` with no plan in hand: the one-off call of the README, which
                makes the plan, its buffers and the pass;
* ``batch``     several volumes of uneven shapes through ``msc.Batch`` as one submission;
* ``static``    the gradient and the critical cells into the caller's own tensors, for programs
                that may not allocate;
* ``arcs``      a pass and what is asked for after it: D* by 2-saddle and the cells along both
                sorts of arc;
* ``host``      a field in pinned host memory copied to the device, a pass, and every output into the
                program's pinned host buffers;
* ``simplify``  a pass and the persistence simplification of its complex at 5 % of the field's
                range.

Every output is a whole number (cell ids, labels, exact path counts, offsets).
"""
import random

import numpy as np
import torch

from paper_2009_03707_gb300 import msc

# Output sizes per voxel of each sort of field, for the bytes that a pass cannot do without:
# critical cells, of which 1-saddles, 2-saddles; D* entries.  They change little with the grid.
DENSITY = {
    "lattice": (0.0008, 0.0004, 0.0002, 0.0007),
    "grf": (0.36, 0.162, 0.108, 0.71),
    "scan": (0.27, 0.121, 0.080, 0.54),
    "blobs": (0.045, 0.021, 0.011, 0.108),
}


def listed():
    return [
        # the smallest call: a coarse, smooth field with a little noise, where latency and launches count
        {"name": "lattice-32", "kind": "compute", "field": "lattice", "nx": 32, "ny": 32, "nz": 32},
        # a small region of interest with odd extents, rough at the voxel scale
        {"name": "grf-61x75x49", "kind": "compute", "field": "grf", "nx": 61, "ny": 75, "nz": 49, "alpha": 3.0},
        # one volume of a collection of uneven shapes, as simulations of odd domains give them
        {"name": "grf-173x97x141", "kind": "compute", "field": "grf", "nx": 173, "ny": 97, "nz": 141, "alpha": 2.5},
        # the headline workload: a 256^3 Gaussian random field, shallow minor, many critical cells
        {"name": "grf-256", "kind": "compute", "field": "grf", "nx": 256, "ny": 256, "nz": 256, "alpha": 3.0},
        # a scanned volume: 8-bit values, so ties and plateaus everywhere
        {"name": "scan-203x256x178", "kind": "compute", "field": "scan", "nx": 203, "ny": 256, "nz": 178, "alpha": 3.5},
        # the largest single volume: smooth blobs under faint noise, long gradient paths, deep minor
        {"name": "blobs-512", "kind": "compute", "field": "blobs", "nx": 512, "ny": 512, "nz": 512},
        # a one-off analysis: no plan in hand
        {"name": "fresh-128", "kind": "fresh", "field": "grf", "nx": 128, "ny": 128, "nz": 128, "alpha": 3.0},
        # several volumes of uneven shapes submitted together
        {"name": "batch-5", "kind": "batch", "field": "grf", "volumes": 5, "lo": 48, "hi": 192, "shapes": 100, "alpha": 2.5},
        # a program whose own pool holds the GPU's memory
        {"name": "static-161x190x133", "kind": "static", "field": "grf", "nx": 161, "ny": 190, "nz": 133, "alpha": 3.0},
        # a pass and the geometry of its arcs, for drawing them or measuring along them
        {"name": "arcs-192x160x144", "kind": "arcs", "field": "grf", "nx": 192, "ny": 160, "nz": 144, "alpha": 3.0},
        # host to host, as a program that reads a time step and writes its complex to a file
        {"name": "host-144x120x167", "kind": "host", "field": "grf", "nx": 144, "ny": 120, "nz": 167, "alpha": 3.0},
        # a noisy field's complex simplified, the usual next step
        {"name": "simplify-256", "kind": "simplify", "field": "grf", "nx": 256, "ny": 256, "nz": 256, "alpha": 3.0},
    ]


def _extents(rng, lo, hi, voxels):
    """Three extents over [lo, hi] on a log scale (odd ones among them), at most `voxels` in all."""
    while True:
        e = [int(round(lo * (hi / lo) ** rng.random())) for _ in range(3)]
        if e[0] * e[1] * e[2] <= voxels:
            return {"nx": e[0], "ny": e[1], "nz": e[2]}


def draw(rng):
    kind = rng.choice(["compute", "compute", "compute", "fresh", "batch", "static", "arcs", "host", "simplify"])
    alpha = round(rng.uniform(2.5, 3.5), 2)
    if kind == "batch":
        return {"kind": kind, "field": "grf", "volumes": rng.randint(2, 5), "lo": 48, "hi": 192,
                "shapes": rng.randint(0, 10 ** 6), "alpha": alpha}
    if kind == "compute":
        field = rng.choice(["lattice", "grf", "grf", "scan", "blobs"])
        return dict({"kind": kind, "field": field, "alpha": alpha}, **_extents(rng, 24, 448, 384 ** 3))
    # blobs are not simplified here: the paths between the deep arcs of some outnumber 64 bits
    field = rng.choice(["grf", "scan"] if kind == "simplify" else ["grf", "scan", "blobs"])
    top = {"fresh": 192, "static": 140, "arcs": 256, "host": 192, "simplify": 168}[kind]
    return dict({"kind": kind, "field": field, "alpha": alpha}, **_extents(rng, 24, 1.5 * top, top ** 3))


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _grf(nz, ny, nx, alpha, gen):
    """White noise shaped to the power spectrum k^-alpha, zero mean, unit deviation, in 64 bits."""
    spec = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64))
    kz = torch.fft.fftfreq(nz, device="cuda", dtype=torch.float64)[:, None, None]
    ky = torch.fft.fftfreq(ny, device="cuda", dtype=torch.float64)[None, :, None]
    kx = torch.fft.rfftfreq(nx, device="cuda", dtype=torch.float64)[None, None, :]
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    k[0, 0, 0] = 1.0
    amp = k ** (-alpha / 2.0)
    amp[0, 0, 0] = 0.0
    f = torch.fft.irfftn(spec * amp, s=(nz, ny, nx))
    return (f - f.mean()) / f.std()


def _blobs(nz, ny, nx, seed, gen):
    """Gaussian blobs of deviation 2..20 voxels, one per 67 thousand voxels, plus N(0, 1e-3) noise."""
    rng = np.random.default_rng(seed)
    n = max(8, round(2000 * nx * ny * nz / 512 ** 3))
    centres = rng.uniform(0.0, 1.0, size=(n, 3)) * np.array([nx, ny, nz])
    sigmas = rng.uniform(2.0, 20.0, size=n)
    amps = rng.uniform(-1.0, 1.0, size=n)
    f = torch.randn((nz, ny, nx), generator=gen, device="cuda") * 1e-3
    ax = [torch.arange(m, device="cuda", dtype=torch.float32) for m in (nx, ny, nz)]
    for c, s, a in zip(centres, sigmas, amps):
        r = [slice(max(0, int(np.ceil(c[d] - 5 * s))), int(np.floor(c[d] + 5 * s)) + 1) for d in range(3)]
        e = [torch.exp(-0.5 * ((ax[d][r[d]] - float(c[d])) / float(s)) ** 2) for d in range(3)]
        f[r[2], r[1], r[0]] += (float(a) * e[2])[:, None, None] * (e[1][:, None] * e[0][None, :])
    return f


def _field(case, dims, seed):
    nx, ny, nz = dims
    gen = _generator(seed)
    sort = case["field"]
    if sort == "lattice":  # a cosine lattice of period 16 with U[0, 1e-3] noise
        t = [torch.cos(2.0 * np.pi * torch.arange(m, device="cuda", dtype=torch.float64) / 16.0) for m in dims]
        f = t[0][None, None, :] + t[1][None, :, None] + t[2][:, None, None]
        f = f + 1e-3 * torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    elif sort == "blobs":
        f = _blobs(nz, ny, nx, seed, gen)
    else:
        f = _grf(nz, ny, nx, case["alpha"], gen)
        if sort == "scan":  # 8-bit values
            f = torch.round((f - f.min()) / (f.max() - f.min()) * 255.0)
    return f.to(torch.float32).contiguous()


def _shapes(case):
    """The extents (nx, ny, nz) of a batch's volumes."""
    rng = random.Random(case["shapes"])
    return [tuple(rng.randint(case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["volumes"])]


# Room of a program's own buffers for the outputs that vary with the field, in entries per voxel.
ROOM = {"compute": {"words": 4, "longs": 2}, "fresh": {"words": 4, "longs": 2}, "batch": {"words": 4, "longs": 2},
        "arcs": {"words": 20, "longs": 6}, "simplify": {"bytes": 1, "words": 6, "longs": 6}}
DTYPE = {"bytes": torch.uint8, "words": torch.int32, "longs": torch.int64}


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "batch":
        state["fields"] = [_field(case, d, seed * 1000 + i) for i, d in enumerate(_shapes(case))]
        state["batch"], state["plans"] = msc.Batch(), None
        n = sum(f.numel() for f in state["fields"])
    else:
        dims = (case["nx"], case["ny"], case["nz"])
        state["field"] = _field(case, dims, seed)
        n = state["field"].numel()
    if kind in ROOM:
        state["packed"] = {k: torch.zeros(r * n + 4096, dtype=DTYPE[k], device="cuda") for k, r in ROOM[kind].items()}
    if kind == "static":
        msc.msc_static_prepare(torch.cuda.current_device())
        state["words"] = torch.zeros(state["field"].shape, dtype=torch.int32, device="cuda").view(torch.uint32)
        # room for as many cells of each dimension as vertices: no field here comes near it
        state["cells"] = [torch.zeros(n, dtype=torch.int32, device="cuda").view(torch.uint32) for _ in range(4)]
        state["capacity"] = [n] * 4
    elif kind not in ("batch", "fresh"):
        state["plan"] = msc.Plan(dims)
    if kind == "host":
        state["host_field"] = state["field"].cpu().pin_memory()
        room = {"cells0": 1, "cells1": 1, "cells2": 1, "cells3": 1, "min_arcs": 2, "max_arcs": 2, "vertex_min": 1,
                "cube_max": 1, "dstar_rowptr": 1, "dstar_col": 2, "dstar_count": 2}
        state["host"] = {k: torch.zeros(r * n + 1024, dtype=DTYPE["longs" if k in ("dstar_rowptr", "dstar_count") else "words"],
                                        pin_memory=True) for k, r in room.items()}
    if kind == "simplify":
        state["threshold"] = 0.05 * float(state["field"].max() - state["field"].min())
    return state


def _packed(state, name, tensors):
    """The tensors one after another in the program's own buffer (a plan's outputs are overwritten by
    its next pass).  The buffer has the same size for every field; what no output reaches stays 0."""
    signed = {torch.uint32: torch.int32, torch.uint64: torch.int64}  # torch has operators for these
    flat = [t.view(signed[t.dtype]).reshape(-1) if t.dtype in signed else t.reshape(-1) for t in tensors]
    torch.cat(flat, out=state["packed"][name][:sum(t.numel() for t in flat)])
    return state["packed"][name]


def _outputs(plan):
    """Every output of the plan's last pass: the labels of every vertex and cube, then the 32-bit and
    the 64-bit ones.  The labels stay in the plan's memory, so they are kept with the plan that owns it."""
    _, cells = msc.msc_critical(plan)
    min_arcs, max_arcs, vertex_min, cube_max = msc.msc_extremum_arcs(plan)
    rowptr, col, count = msc.msc_saddle_arcs(plan)
    labels = [vertex_min.view(torch.int32), cube_max.view(torch.int32)]
    for t in labels:
        t.plan = plan
    return labels, [*cells, min_arcs, max_arcs, col], [rowptr, count]


def run(state):
    kind = state["kind"]
    if kind == "batch":
        ticket, plans = state["batch"].msc_batch_submit(state["fields"], state["plans"])
        status = state["batch"].msc_batch_wait(ticket)
        state["plans"] = plans
        outs = [_outputs(p) for p in plans]
        return {"status": status, "labels": [o[0] for o in outs],
                "words": _packed(state, "words", [t for o in outs for t in o[1]]),
                "longs": _packed(state, "longs", [t for o in outs for t in o[2]])}
    if kind == "static":
        counts = msc.msc_gradient_critical_static(state["field"], state["words"], state["cells"], state["capacity"])
        return {"counts": counts, "words": state["words"].view(torch.int32),
                "cells": [c.view(torch.int32) for c in state["cells"]]}
    if kind == "fresh":
        out = msc.compute(state["field"])
        labels = [out["vertex_min"].view(torch.int32), out["cube_max"].view(torch.int32)]
        for t in labels:
            t.plan = out["plan"]
        words, longs = [*out["cells"], out["min_arcs"], out["max_arcs"], out["dstar"][1]], [out["dstar"][0], out["dstar"][2]]
        return {"counts": out["counts"], "labels": labels, "words": _packed(state, "words", words),
                "longs": _packed(state, "longs", longs)}
    plan = state["plan"]
    if kind == "host":
        state["field"].copy_(state["host_field"], non_blocking=True)
    msc.msc_compute(plan, state["field"])
    if kind == "host":
        sizes = [msc.msc_copy_to_host_into(plan, k, t) for k, t in state["host"].items()]
        return {"sizes": sizes, "host": state["host"]}
    if kind == "simplify":
        out = msc.msc_simplify(plan, state["field"], state["threshold"])
        return {"counts": out["counts"], "rounds": out["n_rounds"], "cancelled": out["n_cancelled"],
                "bytes": _packed(state, "bytes", [out["alive"]]),
                "words": _packed(state, "words", [out["adj"], out["log"]]),
                "longs": _packed(state, "longs", [out["nodeptr"], out["mult"]])}
    labels, words, longs = _outputs(plan)
    if kind == "arcs":
        colptr, row, count = msc.msc_saddle_arcs_csc(plan)
        offsets, cells = msc.msc_arc_geometry(plan)
        ss_offsets, ss_cells = msc.msc_saddle_arc_geometry(plan)
        words += [row, cells, ss_cells]
        longs += [colptr, count, offsets, ss_offsets]
    return {"labels": labels, "words": _packed(state, "words", words), "longs": _packed(state, "longs", longs)}


def work(case):
    """Bytes: the field read once and each output written once (see DENSITY).  Operations: the 26
    comparisons of a vertex with its neighbours that the pairing starts from."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(x * y * z for x, y, z in _shapes(case))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    crit, s1, s2, dstar = (d * n for d in DENSITY[case["field"]])
    adj = 2 * (2 * s1 + 2 * s2 + dstar)  # the 1-skeleton: every arc at both of its ends
    if kind == "static":
        out = 4 * n + 4 * crit
    elif kind == "simplify":
        out = 9 * crit + 12 * adj / 8  # about an eighth of the complex is left
    else:
        out = 4 * crit + 8 * (s1 + s2) + 8 * n + 8 * s1 + 12 * dstar
        if kind == "arcs":
            # offsets and cells: a saddle-extremum arc has about 6 cells, a saddle-saddle arc 8.6
            out += 8 * s2 + 12 * dstar + 2 * (s1 + s2) * (8 + 4 * 6) + dstar * (8 + 4 * 8.6)
    return {"bytes": 4 * n + out, "flops": 26 * n}


def exact(case, seed):
    """Every output is a whole number, which is compared for equality: there is no nearer value."""
    return None
