"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` gives what a user's program has in hand before the call (a context with
its finalized geometry, the device inputs and outputs), ``run`` makes the call through the package's entry points,
``work`` states the bytes and operations the call cannot do without, ``exact`` the outputs in 64 bits from formulas
of its own where the geometry has closed forms.

A context with its geometry (and, for the learned mode, its trained network) is made once per scene and process and
kept, as a program that transports batch after batch keeps it; the track seed, the rays, the queries and the training
samples are new for every seed.
"""
import math

import numpy as np
import torch

import paper_1209_5235_gb300 as g4
import synth
from synth.mlp_init import mlp_init

MODES = {"fp64": g4.G4N_MODE_FP64, "fp32_recheck": g4.G4N_MODE_FP32_RECHECK, "learned": g4.G4N_MODE_LEARNED}
N_BATCHES = 100          # tally rows of a transport, as the benchmark takes
TWO_PI = 2.0 * math.pi


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # a first look at a setup: a small scene, few tracks, every option at its default; launches and latency count
        {"name": "tiny_1e4", "call": "transport", "scene": "tiny", "tracks": 10000, "mode": "fp64"},
        # dose in a sampling calorimeter: box cells, the benchmark's batch on the schedule the tuner picks for it
        {"name": "calorimeter_1e6", "call": "transport", "scene": "calorimeter", "tracks": 1000000, "mode": "fp64",
         "staged": True, "blocks_per_sm": 8},
        # the same scene from a host program: numpy tallies out of host buffers, a batch of odd size, a mid-sized pool
        {"name": "calorimeter_host_2e5", "call": "transport_host", "scene": "calorimeter", "tracks": 200003,
         "mode": "fp64", "staged": True},
        # the benchmark's default line: the barrel detector, ten million tracks, FP32 bounds, staged queues with the
        # relocation kernel
        {"name": "barrel_1e7", "call": "transport", "scene": "barrel", "tracks": 10000000, "mode": "fp32_recheck",
         "staged": True, "reloc": True, "blocks_per_sm": 16},
        # the barrel as a first user calls it: default mode and schedule, per-track hashes and lengths for a comparison
        {"name": "barrel_default_3e5", "call": "transport", "scene": "barrel", "tracks": 300007, "mode": "fp64",
         "per_track": True},
        # a deep hierarchy (32 levels), every level searched on the way up and down
        {"name": "nested_barrel_1e6", "call": "transport", "scene": "nested_barrel", "tracks": 1000000,
         "mode": "fp32_recheck", "staged": True, "reloc": True},
        # many independent geometries of uneven size in one launch: random boxes, tubes and orbs, FP32 bounds
        {"name": "batched_worlds_48", "call": "transport", "scene": "batched", "worlds": 48, "scale": 0.5,
         "mode": "fp32_recheck", "block_size": 64, "walk_budget": 65536},
        # the learned proposal where it pays: plates listed farthest first, the network inside the step kernel
        {"name": "stack_learned_1e6", "call": "transport", "scene": "stack", "tracks": 1000000, "mode": "learned",
         "staged": True, "drain": -1},
        # which volume holds each point: hit maps and dose grids, ten million points
        {"name": "locate_barrel_1e7", "call": "locate", "scene": "barrel", "n": 10000000},
        # distance, safety and limiter for an external stepping loop
        {"name": "compute_step_barrel_1e6", "call": "compute_step", "scene": "barrel", "n": 1000003,
         "mode": "fp32_recheck"},
        # the paper's own benchmark: free paths through the 8000 balls, random rays
        {"name": "free_path_random_1e5", "call": "free_path", "rays": "random", "n": 100000, "mode": "fp64"},
        # training the proposal network, one epoch of a logged sample set
        {"name": "mlp_train_1e6", "call": "mlp_train", "n": 1048576, "batch": 4096, "epochs": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["transport"] * 5 + ["transport_host", "locate", "compute_step", "free_path", "mlp_train"])
    if call in ("transport", "transport_host"):
        scene = rng.choice(["tiny", "calorimeter", "barrel", "nested_barrel", "batched", "stack"])
        mode = rng.choice(["fp64", "fp32_recheck"] + (["learned"] if scene == "stack" else []))
        c = {"call": call, "scene": scene, "mode": mode}
        if scene == "batched":
            c["worlds"] = rng.randint(8, 48)
            c["scale"] = round(rng.uniform(0.05, 0.5), 3)
        else:
            c["tracks"] = _log_int(rng, 1000, 3000000 if scene in ("calorimeter", "stack", "tiny") else 2000000)
        if rng.random() < 0.6 and scene != "batched":
            c["staged"] = True
            if scene in ("barrel", "nested_barrel") and rng.random() < 0.7:
                c["reloc"] = True
        if call == "transport" and rng.random() < 0.3:
            c["per_track"] = True
        return c
    if call == "locate":
        return {"call": call, "scene": rng.choice(["calorimeter", "barrel"]), "n": _log_int(rng, 1000, 10000000)}
    if call == "compute_step":
        return {"call": call, "scene": rng.choice(["calorimeter", "barrel"]), "n": _log_int(rng, 1000, 2000000),
                "mode": rng.choice(["fp64", "fp32_recheck"])}
    if call == "free_path":
        return {"call": call, "rays": "random", "n": _log_int(rng, 1000, 400000),
                "mode": rng.choice(["fp64", "fp32_recheck"])}
    batch = 16 * _log_int(rng, 16, 512)
    return {"call": call, "n": batch * rng.randint(8, 256) + rng.randint(0, 15), "batch": batch, "epochs": 1}


# ---------------------------------------------------------------- what a program keeps

_kept = {}


def _scene(case):
    name, sc = case["scene"], synth.scenes
    if name == "tiny":
        return sc.tiny_scene(), sc.tiny_source()
    if name == "calorimeter":
        return sc.calorimeter_scene(voxel=sc.VoxelSpec(mode="smart")), sc.calorimeter_source()
    if name == "barrel":
        return sc.barrel_scene(), sc.barrel_source()
    if name == "nested_barrel":
        return sc.nested_barrel_scene(), sc.barrel_source()
    if name == "stack":
        return sc.reversed_stack_scene(), sc.reversed_stack_source()
    return sc.spheres_scene(), None


def _context(case):
    """(context, geometry ids, scenes, source) of the case's scene, made once per process."""
    key = (case.get("scene"), case.get("worlds"))
    if key in _kept:
        return _kept[key]
    ctx = g4.g4n_create(0)
    if case["scene"] == "batched":
        pairs = synth.scenes.batched_scenes(case["worlds"], d_range=(10, 2000))
        got = (ctx, [g4.build_scene(ctx, s) for s, _ in pairs], pairs, synth.scenes.batched_source())
    else:
        scene, source = _scene(case)
        got = (ctx, [g4.build_scene(ctx, scene)], [(scene, 0)], source)
        if case["scene"] == "stack":  # the network, trained on steps that the plain navigator logs
            items = g4.make_items([(got[1][0], 200000, 50_000_000, source, 0)])
            samples = g4.g4n_mlp_log(ctx, items, 0x7A0C0027, 1_000_000, scene.n_volumes + 2)
            g4.g4n_mlp_load(ctx, mlp_init(15))
            g4.g4n_mlp_train(ctx, *samples, epochs=2, batch=2048, lr=2e-3, seed=6)
    _kept[key] = got
    return got


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _isotropic(n, gen):
    d = torch.randn((3, n), dtype=torch.float64, device="cuda", generator=gen)
    return (d / d.square().sum(0).sqrt()).contiguous()


def _queries(case, seed):
    """Points uniform in the scene's query box, isotropic directions, a physics proposal ~ Exp(100 mm)."""
    gen = _generator(seed)
    lo, hi = (torch.tensor(b, dtype=torch.float64, device="cuda") for b in synth.scenes.QUERY_BOXES[case["scene"]])
    pos = torch.rand((3, case["n"]), dtype=torch.float64, device="cuda", generator=gen)
    pos = (lo[:, None] + (hi - lo)[:, None] * pos).contiguous()
    direction = _isotropic(case["n"], gen)
    proposed = torch.empty(case["n"], dtype=torch.float64, device="cuda").exponential_(0.01, generator=gen)
    return pos, direction, proposed


def _rays(case, seed):
    """Rays from the centre of the balls: isotropic, Y ~ Exp(1)."""
    gen = _generator(seed)
    pos = torch.zeros((3, case["n"]), dtype=torch.float64, device="cuda")
    direction = _isotropic(case["n"], gen)
    y = torch.empty(case["n"], dtype=torch.float64, device="cuda").exponential_(1.0, generator=gen)
    return pos, direction, y


def _samples(case, seed):
    """Training samples as the navigator logs them: the point in its node, the direction, log E, the candidate count,
    1; the label is the slot that the ray meets first in a node sliced along z."""
    gen, n = _generator(seed), case["n"]
    point = 2.0 * torch.rand((n, 3), device="cuda", generator=gen) - 1.0
    direction = _isotropic(n, gen).T.float()
    log_e = torch.rand(n, device="cuda", generator=gen)
    ncand = torch.randint(2, 33, (n,), device="cuda", generator=gen, dtype=torch.int32)
    at = (0.5 * (point[:, 2] + 1.0) * ncand).floor() + torch.where(direction[:, 2] > 0, 1.0, -1.0)
    label = torch.minimum(at.clamp(min=0.0).int(), ncand - 1)
    feat = torch.cat([point, direction, log_e[:, None], ncand[:, None] / 32.0, torch.ones((n, 1), device="cuda")], 1)
    return feat.float().contiguous(), label.contiguous(), ncand


def prepare(case, seed):
    call = case["call"]
    if call == "mlp_train":
        if "train" not in _kept:
            _kept["train"] = g4.g4n_create(0)
        return {"case": case, "ctx": _kept["train"], "params": mlp_init(41), "samples": _samples(case, seed)}
    if call == "free_path":
        ctx, gids, _, _ = _context({"scene": "spheres"})
        n = case["n"]
        return {"case": case, "ctx": ctx, "geom": gids[0], "rays": _rays(case, seed),
                "T": torch.empty(n, dtype=torch.float64, device="cuda"),
                "steps": torch.empty(n, dtype=torch.int32, device="cuda")}
    ctx, gids, scenes, source = _context(case)
    if call in ("locate", "compute_step"):
        n = case["n"]
        pos, direction, proposed = _queries(case, seed)
        depth = torch.empty(n, dtype=torch.int32, device="cuda")
        path = torch.empty((g4.G4N_DMAX, n), dtype=torch.int32, device="cuda")
        state = {"case": case, "ctx": ctx, "geom": gids[0], "pos": pos, "dir": direction, "depth": depth, "path": path}
        if call == "compute_step":
            g4.g4n_locate(ctx, gids[0], pos, direction, out_depth=depth, out_path=path)
            state["proposed"] = proposed
            state["out"] = (torch.empty(n, dtype=torch.float64, device="cuda"),
                            torch.empty(n, dtype=torch.float64, device="cuda"),
                            torch.empty(n, dtype=torch.int32, device="cuda"))
        return state
    entries, column, first = [], 0, 0
    for gid, (scene, tracks) in zip(gids, scenes):
        n = case["tracks"] if "tracks" in case else max(1, int(tracks * case["scale"]))
        entries.append((gid, n, first, source, column))
        column += scene.n_volumes + 2
        first += n
    options = {"mode": MODES[case["mode"]], "block_size": case.get("block_size", 0),
               "blocks_per_sm": case.get("blocks_per_sm", 0), "walk_budget": case.get("walk_budget", 0),
               "drain_tracks": case.get("drain", 0), "n_batches": N_BATCHES,
               "schedule": g4.G4N_SCHEDULE_STAGED if case.get("staged") else g4.G4N_SCHEDULE_PERSISTENT,
               "staged_flags": g4.G4N_STAGED_RELOCATION_KERNEL if case.get("reloc") else 0}
    state = {"case": case, "ctx": ctx, "items": g4.make_items(entries), "seed": seed, "options": options,
             "columns": column}
    if call == "transport":
        state["edep"] = torch.zeros((N_BATCHES, column), dtype=torch.float64, device="cuda")
        state["counters"] = torch.zeros(g4.G4N_N_COUNTERS, dtype=torch.int64, device="cuda")
        if case.get("per_track"):
            state["hash"] = torch.zeros(first, dtype=torch.int64, device="cuda")
            state["length"] = torch.zeros(first, dtype=torch.float64, device="cuda")
    return state


# ---------------------------------------------------------------- the calls

def run(state):
    case, ctx = state["case"], state["ctx"]
    call = case["call"]
    if call == "transport":
        state["edep"].zero_()
        state["counters"].zero_()
        g4.g4n_transport_batch(ctx, state["items"], state["seed"], state["edep"], state["counters"],
                               track_hash=state.get("hash"), track_len=state.get("length"), **state["options"])
        return [state[k] for k in ("edep", "counters", "hash", "length") if k in state]
    if call == "transport_host":
        out = g4.g4n_transport_batch_host(ctx, state["items"], state["seed"], state["columns"], **state["options"])
        return [out["edep"], out["counters"].view(np.int64)]
    if call == "locate":
        return list(g4.g4n_locate(ctx, state["geom"], state["pos"], state["dir"], out_depth=state["depth"],
                                  out_path=state["path"]))
    if call == "compute_step":
        return list(g4.g4n_compute_step(ctx, state["geom"], state["pos"], state["dir"], state["depth"], state["path"],
                                        proposed=state["proposed"], mode=MODES[case["mode"]], out=state["out"]))
    if call == "free_path":
        pos, direction, y = state["rays"]
        return list(g4.g4n_free_path(ctx, state["geom"], pos, direction, y, synth.scenes.SPHERES_ENERGY,
                                     mode=MODES[case["mode"]], out_T=state["T"], out_steps=state["steps"]))
    g4.g4n_mlp_load(ctx, state["params"])
    losses = g4.g4n_mlp_train(ctx, *state["samples"], epochs=case["epochs"], batch=case["batch"], lr=2e-3, seed=5)
    return [g4.g4n_mlp_get(ctx), losses]


# ---------------------------------------------------------------- work

# volumes, and steps and interactions per track, of the transport scenes (counted by the library's own counters)
SCENES = {"tiny": (11, 5.6, 4.2), "calorimeter": (5002, 19.1, 2.3), "barrel": (3951, 9.6, 3.0),
          "nested_barrel": (3951, 9.9, 3.0), "batched": (280, 4.0, 3.5), "stack": (25, 17.4, 0.9)}
FLOPS_STEP, FLOPS_INTERACT = 150, 60   # add, multiply, compare: 1; fused, divide, root: 2


def work(case):
    call = case["call"]
    if call in ("transport", "transport_host"):
        volumes, steps, inter = SCENES[case["scene"]]
        worlds = case.get("worlds", 1)
        # the batched worlds have 10^3 to 10^5 tracks each, spread over their logarithm: 21.5 thousand in the mean
        n = case.get("tracks") or int(worlds * 21500 * case["scale"])
        out = 2 * 8 * N_BATCHES * worlds * (volumes + 2) + 8 * g4.G4N_N_COUNTERS + (16 * n if case.get("per_track") else 0)
        return {"bytes": out, "flops": n * (steps * FLOPS_STEP + inter * FLOPS_INTERACT)}
    n = case["n"]
    if call == "locate":    # point and direction in; depth and path out
        return {"bytes": n * (48 + 4 + 4 * g4.G4N_DMAX), "flops": n * 150}
    if call == "compute_step":   # point, direction, depth, leaf, proposal in; step, safety, limiter out
        return {"bytes": n * (48 + 4 + 4 + 8 + 8 + 8 + 4), "flops": n * 300}
    if call == "free_path":
        return {"bytes": n * (48 + 8 + 8 + 4), "flops": n * 2.4 * 150}
    used = case["epochs"] * (n // case["batch"]) * case["batch"]
    return {"bytes": used * (36 + 4 + 4) + 3 * 4 * g4.G4N_MLP_N_PARAMS,
            "flops": used * 6 * (9 * 64 + 64 * 64 + 64 * 32)}


# ---------------------------------------------------------------- exact outputs, in 64 bits

def exact(case, seed):
    call = case["call"]
    if call == "free_path":
        return [_exact_free_path(case, seed), None]
    if call == "compute_step":
        return [(_exact_barrel_step if case["scene"] == "barrel" else _exact_calorimeter_step)(case, seed), None, None]
    if call == "mlp_train":
        return _exact_training(case, seed)
    return None  # a history is as long as its random numbers make it; a located volume is no computed number


def _roots(b, c):
    """Both roots of t^2 + 2 b t + c, NaN where there are none."""
    q = -(b + torch.copysign((b * b - c).sqrt(), b))
    return torch.minimum(q, c / q), torch.maximum(q, c / q)


def _exact_free_path(case, seed):
    scene, _ = _scene({"scene": "spheres"})
    _, direction, y = _rays(case, seed)
    centres = torch.tensor([p.t for p in scene.placements[1:]], dtype=torch.float64, device="cuda")
    radius = scene.solids[1].params[0]
    mu = scene.materials[1].mu_compton[0] + scene.materials[1].mu_photo[0]
    c = centres.square().sum(1) - radius * radius
    out = []
    for k in range(0, case["n"], 8192):
        lo, hi = _roots(-(direction[:, k:k + 8192].T @ centres.T), c[None, :])
        lo = torch.where((lo > 0.0) & ~lo.isnan(), lo, math.inf)
        lo, at = lo.sort(dim=1)
        lo, at = lo[:, :64], at[:, :64]
        chord = torch.where(lo.isinf(), 0.0, hi.gather(1, at) - lo)
        depth = torch.cumsum(chord, 1) * mu
        before = depth - chord * mu
        yk = y[k:k + 8192, None]
        t = torch.where((depth >= yk) & ~lo.isinf(), lo + (yk - before) / mu, math.inf)
        out.append(t.min(dim=1).values)
    return torch.cat(out)


def _first(*ts):
    """The smallest of the distances that are positive numbers."""
    return torch.stack([torch.where(t > 0.0, t, math.inf) for t in ts]).min(dim=0).values


def _box_exit(p, u, half):
    return ((torch.copysign(half, u) - p) / u).min(dim=0).values


def _exact_calorimeter_step(case, seed):
    p, u, proposed = _queries(case, seed)
    depth = 375.0
    edges = torch.tensor(np.concatenate([[0.0], np.cumsum([5.0, 10.0] * 25)]), device="cuda")
    inside = (p[0].abs() < 500.0) & (p[1].abs() < 500.0) & (p[2] > 0.0) & (p[2] < depth)
    layer = (torch.bucketize(p[2].contiguous(), edges, right=True) - 1).clamp(0, 49)
    lo, hi = edges[layer], edges[layer + 1]
    centre = torch.stack([(p[0] / 100.0).floor() * 100.0 + 50.0, (p[1] / 100.0).floor() * 100.0 + 50.0, 0.5 * (lo + hi)])
    half = torch.stack([torch.full_like(lo, 50.0), torch.full_like(lo, 50.0), 0.5 * (hi - lo)])
    cell = _box_exit(p - centre, u, half)
    world = _box_exit(p, u, torch.full_like(p, 1000.0))
    q = p - torch.tensor([0.0, 0.0, 0.5 * depth], device="cuda", dtype=torch.float64)[:, None]
    env = torch.tensor([500.0, 500.0, 0.5 * depth], device="cuda", dtype=torch.float64)[:, None].expand_as(q)
    a, b = (-env - q) / u, (env - q) / u
    t_in, t_out = torch.minimum(a, b).max(dim=0).values, torch.maximum(a, b).min(dim=0).values
    world = torch.where((t_out > t_in) & (t_in > 0.0), torch.minimum(world, t_in), world)
    return torch.minimum(torch.where(inside, cell, world), proposed)


def _exact_barrel_step(case, seed):
    scene, _ = _scene({"scene": "barrel"})
    pos, direction, proposed = _queries(case, seed)
    r_in, r_out, half_z, shells, segments = 50.0, 1500.0, 1500.0, 30, 64
    dr, dphi = (r_out - r_in) / shells, TWO_PI / segments
    centres, radii = [], []
    for pl in scene.placements:
        solid = scene.solids[pl.solid]
        if solid.kind == synth.scenes.ORB:  # placed in a segment that is rotated about z
            c, s = scene.placements[pl.mother].rot
            centres.append((c * pl.t[0] - s * pl.t[1], s * pl.t[0] + c * pl.t[1], pl.t[2]))
            radii.append(solid.params[0])
    centres = torch.tensor(centres, dtype=torch.float64, device="cuda")
    radii = torch.tensor(radii, dtype=torch.float64, device="cuda")
    out = []
    for k in range(0, case["n"], 65536):
        p, u = pos[:, k:k + 65536], direction[:, k:k + 65536]
        b = (p * u).sum(0)[:, None] - u.T @ centres.T
        gap = p[:, None, :] - centres.T[:, :, None]
        lo, hi = _roots(b, gap.square().sum(0).T - radii.square()[None, :])
        within = (lo < 0.0) & (hi > 0.0)
        orb_exit = torch.where(within, hi, math.inf).min(dim=1).values
        orb_entry = torch.where(lo > 0.0, lo, math.inf).min(dim=1).values
        a, bb, r2 = u[:2].square().sum(0), (p[:2] * u[:2]).sum(0), p[:2].square().sum(0)
        r = r2.sqrt()
        shell = ((r - r_in) / dr).floor().clamp(0, shells - 1)

        def cylinder(radius):
            c = r2 - radius * radius
            return _roots(bb / a, c / a)

        to_z = (torch.copysign(torch.full_like(r, half_z), u[2]) - p[2]) / u[2]
        seg = (torch.atan2(p[1], p[0]) / dphi).floor()
        planes = []
        for side, sign in ((seg, 1.0), (seg + 1.0, -1.0)):  # towards each phi plane, from its inner side
            c, s = torch.cos(side * dphi), torch.sin(side * dphi)
            dist, speed = sign * (c * p[1] - s * p[0]), -sign * (c * u[1] - s * u[0])
            planes.append(torch.where(speed > 0.0, dist / speed, math.inf))
        rmin, rmax = cylinder(r_in + shell * dr), cylinder(r_in + (shell + 1.0) * dr)
        segment = _first(to_z, rmin[0], rmax[1], *planes, orb_entry)
        # outside the shells: into their common envelope, or out of the world
        inner, outer = cylinder(torch.full_like(r, r_in)), cylinder(torch.full_like(r, r_out))
        caps = (torch.where(u[2] < 0.0, half_z, -half_z) - p[2]) / u[2]
        at = (p[:2] + caps * u[:2]).square().sum(0)
        caps = torch.where((at > r_in * r_in) & (at < r_out * r_out), caps, math.inf)
        inner = torch.where((p[2] + inner[1] * u[2]).abs() < half_z, inner[1], math.inf)
        outer = torch.where((r > r_out) & ((p[2] + outer[0] * u[2]).abs() < half_z), outer[0], math.inf)
        world = _first(_box_exit(p, u, torch.full_like(p, 2000.0)), caps, inner, outer)
        in_shell = (r > r_in) & (r < r_out) & (p[2].abs() < half_z)
        t = torch.where(in_shell, segment, world)
        out.append(torch.minimum(torch.where(within.any(dim=1), orb_exit, t), proposed[k:k + 65536]))
    return torch.cat(out)


def _exact_training(case, seed):
    """The documented training in 64 bits: minibatches of a fixed-stride permutation, masked softmax cross-entropy,
    Adam (0.9, 0.999, 1e-8)."""
    feat, label, ncand = _samples(case, seed)
    n, batch, wrap = case["n"], case["batch"], (1 << 64) - 1
    packed, parts, at = torch.tensor(mlp_init(41), dtype=torch.float64, device="cuda"), [], 0
    for shape in ((9, 64), (64,), (64, 64), (64,), (64, 32), (32,)):
        size = math.prod(shape)
        parts.append(packed[at:at + size].reshape(shape).clone().requires_grad_())
        at += size
    m, v = [torch.zeros_like(x) for x in parts], [torch.zeros_like(x) for x in parts]
    losses, step = [], 0
    for epoch in range(case["epochs"]):
        h = (5 * 0x9E3779B97F4A7C15 + epoch * 0xD1B54A32D192ED03 + 1) & wrap
        h ^= h >> 31
        h = (h * 0xBF58476D1CE4E5B9) & wrap
        h ^= h >> 27
        stride = (h % n) | 1
        while math.gcd(stride, n) != 1:
            stride += 2
        offset, total = (h >> 17) % n, 0.0
        for k in range(n // batch):
            rows = (torch.arange(k * batch, (k + 1) * batch, device="cuda") * stride + offset) % n
            w1, b1, w2, b2, w3, b3 = parts
            x = torch.nn.functional.gelu(feat[rows].double() @ w1 + b1)
            x = torch.nn.functional.gelu(x @ w2 + b2) @ w3 + b3
            x = x.masked_fill(torch.arange(32, device="cuda")[None, :] >= ncand[rows, None], -math.inf)
            loss = torch.nn.functional.cross_entropy(x, label[rows].long())
            grads = torch.autograd.grad(loss, parts)
            total, step = total + float(loss), step + 1
            with torch.no_grad():
                for x, g, mm, vv in zip(parts, grads, m, v):
                    mm.mul_(0.9).add_(g, alpha=0.1)
                    vv.mul_(0.999).add_(g * g, alpha=0.001)
                    x -= 2e-3 * (mm / (1 - 0.9 ** step)) / ((vv / (1 - 0.999 ** step)).sqrt() + 1e-8)
        losses.append(total / (n // batch))
    return [torch.cat([x.detach().reshape(-1) for x in parts]), torch.tensor(losses, dtype=torch.float64)]
