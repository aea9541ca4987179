"""The relocation portals, decided on the host for whole faces, against the oracle's search at points of those faces:
every box, tube segment and orb of several scenes, leaving and entering, crossing directions drawn at random."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth
import paper_1209_5235_gb300 as g4
from gpu_common import mixed_scene

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NONE = -2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("portal") / "portal.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(ROOT, "tests", "portal_host.cpp"),
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1209_5235_gb300", "csrc")],
                   check=True)
    return ctypes.CDLL(so)


def portals(lib, scene):
    ctx = g4.g4n_create(-1)
    try:
        gid = g4.build_scene(ctx, scene)
        n = lib.portals_of(ctx, gid, None)
        out = np.zeros(n, dtype=np.int32)
        lib.portals_of.restype = ctypes.c_longlong
        lib.portals_of(ctx, gid, out.ctypes.data_as(ctypes.c_void_p))
    finally:
        g4.g4n_destroy(ctx)
    return out.reshape(-1, 2, 6)


def world_frames(scene):
    frames = []
    for p in scene.placements:
        c, s = p.rot
        if p.mother < 0:
            frames.append((np.array(p.t, dtype=float), c, s))
        else:
            t, mc, ms = frames[p.mother]
            frames.append((t + np.array([mc * p.t[0] - ms * p.t[1], ms * p.t[0] + mc * p.t[1], p.t[2]]),
                           mc * c - ms * s, ms * c + mc * s))
    return frames


def face_point(rng, kind, q, face, edge):
    """A point of the face at least `edge` from the solid's other faces and the outward normal there (None: no such face)."""
    def between(lo, hi):
        return rng.uniform(lo + edge, hi - edge) if hi - lo > 2 * edge else None
    if kind == 0:
        axis, side = face >> 1, 1.0 if face & 1 else -1.0
        p, n = [between(-h, h) for h in q], np.zeros(3)
        p[axis], n[axis] = side * q[axis], side
        return None if None in p else (np.array(p), n)
    if kind == 2:
        n = rng.normal(size=3)
        n /= np.linalg.norm(n)
        return (q[0] * n, n) if face == 0 else None
    rmin, rmax, hz, sphi, dphi = q
    seg = dphi < 2 * math.pi - 1e-12
    if face == 3 and rmin == 0.0 or face >= 4 and not seg:
        return None
    r = rmax if face == 2 else rmin if face == 3 else between(rmin, rmax)
    if r is None:
        return None
    margin = math.asin(min(1.0, 1.01 * edge / r)) if seg else 0.0
    if face >= 4:
        phi = sphi if face == 4 else sphi + dphi
    elif dphi <= 2 * margin:
        return None
    else:
        phi = rng.uniform(sphi + margin, sphi + dphi - margin)
    z = (hz if face == 1 else -hz) if face < 2 else between(-hz, hz)
    if z is None:
        return None
    n = {0: (0, 0, -1), 1: (0, 0, 1), 2: (math.cos(phi), math.sin(phi), 0), 3: (-math.cos(phi), -math.sin(phi), 0),
         4: (math.sin(phi), -math.cos(phi), 0), 5: (-math.sin(phi), math.cos(phi), 0)}[face]
    return np.array([r * math.cos(phi), r * math.sin(phi), z]), np.array(n, dtype=float)


SCENES = {"tiny": (synth.scenes.tiny_scene, 0.9),
          "calorimeter": (lambda: synth.scenes.calorimeter_scene(nx=4, ny=4, n_layers=6, voxel=synth.scenes.VoxelSpec()), 0.9),
          "barrel": (lambda: synth.scenes.barrel_scene(n_shells=6, n_phi=16, n_orbs=60, r_out=500.0, half_len=300.0), 0.9),
          "nested barrel": (lambda: synth.scenes.nested_barrel_scene(n_shells=5, n_phi=12, n_orbs=40, r_out=600.0, half_len=300.0), 0.7),
          "mixed": (lambda: mixed_scene(seed=3, n=120, half=300.0), 0.5),
          "spheres": (lambda: synth.scenes.spheres_scene(n_side=4), 0.9),
          "stack": (synth.scenes.reversed_stack_scene, 0.9)}


@pytest.mark.parametrize("name", SCENES)
def test_portals_are_the_oracles_relocation(lib, name):
    make, share = SCENES[name]
    scene = make()
    table, frames = portals(lib, scene), world_frames(scene)
    rng = np.random.default_rng(11)
    pos, dirs, want, faces, have = [], [], [], 0, 0
    for v, pl in enumerate(scene.placements):
        solid = scene.solids[pl.solid]
        if solid.kind == 3:
            assert np.all(table[v] == NONE)
            continue
        for face in range(6):
            for entering in (0, 1):
                leaf = table[v, entering, face]
                at = face_point(rng, solid.kind, solid.params, face, 0.01)
                if at is None:
                    continue
                faces += v > 0
                if leaf == NONE:
                    continue
                have += v > 0
                for _ in range(3):
                    p, n = face_point(rng, solid.kind, solid.params, face, 0.01)
                    d = rng.normal(size=3)
                    d /= np.linalg.norm(d)
                    if abs(d @ n) < 0.01:
                        continue
                    if (d @ n > 0) == bool(entering):
                        d = -d
                    t, c, s = frames[v]
                    turn = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])
                    pos.append(turn @ p + t)
                    dirs.append(turn @ d)
                    want.append(leaf)
    assert faces == 0 or have >= share * faces, (have, faces)
    depth, path = oracle.Geometry(scene).locate_many(np.array(pos), np.array(dirs))
    got = np.where(depth > 0, path[np.arange(len(depth)), np.maximum(depth, 1) - 1], -1)
    bad = np.nonzero(got != np.array(want))[0]
    assert bad.size == 0, (len(want), bad.size, [(pos[i], dirs[i], want[i], got[i]) for i in bad[:3]])


def gap_scene(gap):
    """Solids a gap apart: two boxes, two shells, two segments of a shell, a box on a tube; once about z turned."""
    from synth.scenes import BOX, TUBE, Placement, Scene, Solid, VoxelSpec
    base = synth.scenes.tiny_scene()
    r, w = 100.0, 2 * math.pi
    solids = [Solid(BOX, (500.0, 500.0, 500.0)), Solid(BOX, (20.0, 30.0, 40.0)), Solid(TUBE, (0.0, 50.0, 60.0, 0.0, w)),
              Solid(TUBE, (50.0 + gap, r, 60.0, 0.0, w)), Solid(TUBE, (r + gap, 150.0, 60.0, 0.3, 1.0)),
              Solid(TUBE, (r + gap, 150.0, 60.0, 1.3 + gap / r, 1.0)), Solid(BOX, (30.0, 30.0, 10.0))]
    c, s = math.cos(0.4), math.sin(0.4)
    places = [Placement(-1, 0, 0, (0.0, 0.0, 0.0)), Placement(0, 1, 0, (300.0, 200.0, 0.0)),
              Placement(0, 1, 0, (340.0 + gap, 200.0, 0.0)),
              Placement(0, 1, 0, (-300.0, 200.0, 0.0), (c, s)),
              Placement(0, 1, 0, (-300.0 + c * (40.0 + gap), 200.0 + s * (40.0 + gap), 0.0), (c, s)),
              Placement(0, 2, 0, (0.0, 0.0, 0.0)), Placement(0, 3, 0, (0.0, 0.0, 0.0)), Placement(0, 4, 0, (0.0, 0.0, 0.0)),
              Placement(0, 5, 0, (0.0, 0.0, 0.0)), Placement(0, 6, 0, (0.0, 0.0, 70.0 + gap), (c, s))]
    return Scene("gaps", base.materials, solids, places, VoxelSpec(mode="smart"))


@pytest.mark.parametrize("scale", [1e3, 1e5, 1e6])
@pytest.mark.parametrize("part", [0.2, 0.45, 0.7, 3.0])
def test_portals_know_the_tolerance(lib, scale, part):
    """Across a gap that is a part of the tolerance 1e-9 mm x scale the far solid's band may hold the crossing point, where the
    direction decides: with and without the gap in the band a portal is the oracle's relocation."""
    tol = 1e-9 * scale
    scene = gap_scene(part * tol)
    ctx = g4.g4n_create(-1)
    oracle.set_scale(scale)
    try:
        g4.g4n_set_tolerance_scale(ctx, scale)
        gid = g4.build_scene(ctx, scene)
        n = lib.portals_of(ctx, gid, None)
        table = np.zeros(n, dtype=np.int32)
        lib.portals_of(ctx, gid, table.ctypes.data_as(ctypes.c_void_p))
        table, frames = table.reshape(-1, 2, 6), world_frames(scene)
        rng = np.random.default_rng(12)
        pos, dirs, want = [], [], []
        for v, pl in enumerate(scene.placements):
            solid = scene.solids[pl.solid]
            for face in range(6):
                for entering in (0, 1):
                    if table[v, entering, face] == NONE or face_point(rng, solid.kind, solid.params, face, 0.01) is None:
                        continue
                    for _ in range(20):
                        p, nrm = face_point(rng, solid.kind, solid.params, face, 0.01)
                        d = rng.normal(size=3)
                        d /= np.linalg.norm(d)
                        if abs(d @ nrm) < 0.01:
                            continue
                        if (d @ nrm > 0) == bool(entering):
                            d = -d
                        t, c, s = frames[v]
                        turn = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])
                        pos.append(turn @ p + t)
                        dirs.append(turn @ d)
                        want.append(table[v, entering, face])
        depth, path = oracle.Geometry(scene).locate_many(np.array(pos), np.array(dirs))
        got = np.where(depth > 0, path[np.arange(len(depth)), np.maximum(depth, 1) - 1], -1)
        bad = np.nonzero(got != np.array(want))[0]
        assert len(want) > 100 and bad.size == 0, (len(want), bad.size, [(pos[i], dirs[i], want[i], got[i]) for i in bad[:3]])
    finally:
        oracle.set_scale(1.0)
        g4.g4n_destroy(ctx)
