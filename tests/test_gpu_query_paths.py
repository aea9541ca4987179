"""Query kernels at the sizes where they change their way of working: compute_step answers large batches in tiles sorted
by the kind of the leaf, free paths refill their warps eight lanes at a time.  Every query is independent of the others,
so a large call has to give bit for bit what small calls give for the same queries."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1209_5235_gb300 import build
    build.build()
    import paper_1209_5235_gb300 as g4
    ctx = g4.g4n_create(0)
    yield g4, torch, ctx
    g4.g4n_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("extra", [-1, 0, 1, 511, 513])
def test_compute_step_sorted_tiles(env, mode, extra):
    g4, torch, ctx = env
    gid = g4.build_scene(ctx, synth.scenes.barrel_scene(n_shells=5, n_phi=8, n_orbs=30))
    n = torch.cuda.get_device_properties(0).multi_processor_count * 12 * 512 + extra
    p, v = synth.scenes.query_points("barrel", n, 31)
    v[:, 7] = 2.0   # not a unit direction: refused in the same way wherever the query is sorted to
    T = lambda a: torch.tensor(a, device="cuda")
    pos, dirs = T(p), T(v)
    prop = T(np.random.default_rng(32).exponential(100.0, n))
    depth, path = g4.g4n_locate(ctx, gid, pos, dirs)
    try:
        g4.g4n_sync(ctx)
    except g4.G4NError:
        pass
    whole = g4.g4n_compute_step(ctx, gid, pos, dirs, depth, path, proposed=prop, mode=mode)
    with pytest.raises(g4.G4NError):
        g4.g4n_sync(ctx)
    at = 0
    while at < n:
        k = min(200000, n - at)
        s = slice(at, at + k)
        part = g4.g4n_compute_step(ctx, gid, pos[:, s].contiguous(), dirs[:, s].contiguous(), depth[s].contiguous(),
                                   path[:, s].contiguous(), proposed=prop[s].contiguous(), mode=mode)
        for a, b in zip(whole, part):
            a, b = a[s].cpu().numpy(), b.cpu().numpy()
            assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f")
        at += k
    try:
        g4.g4n_sync(ctx)
    except g4.G4NError:
        pass


@pytest.mark.parametrize("n", [1, 7, 33, 1000, 70001])
def test_free_path_refills(env, n):
    g4, torch, ctx = env
    gid = g4.build_scene(ctx, synth.scenes.spheres_scene(n_side=6))
    _, d, y = synth.scenes.spheres_rays("random", n, seed=41)
    pos = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    dirs = torch.tensor(np.ascontiguousarray(d.T), device="cuda")
    Y = torch.tensor(y, device="cuda")
    T, steps = g4.g4n_free_path(ctx, gid, pos, dirs, Y, 1.0)
    g4.g4n_sync(ctx)
    keep = [0, n // 2, n - 1]
    for k in keep:
        t1, s1 = g4.g4n_free_path(ctx, gid, pos[:, k:k + 1].contiguous(), dirs[:, k:k + 1].contiguous(),
                                  Y[k:k + 1].contiguous(), 1.0)
        assert t1.item() == T[k].item() and s1.item() == steps[k].item()
    assert not torch.isnan(T).any()


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("n", [3001, 1000001])
def test_compute_step_proposals_at_the_ends(env, mode, n):
    """A NaN of either sign and +inf limit nothing: the answers without a proposal, bit for bit.  Zeros, negative values, the
    smallest doubles and -inf come before every boundary: the step is the proposal.  1e300 (beyond any float) limits nothing.
    The larger n takes the sorted tiles."""
    g4, torch, ctx = env
    from synth.mlp_init import mlp_init
    g4.g4n_mlp_load(ctx, mlp_init(3))
    gid = g4.build_scene(ctx, synth.scenes.barrel_scene(n_shells=5, n_phi=8, n_orbs=30))
    p, v = synth.scenes.query_points("barrel", n, 33)
    pos, dirs = torch.tensor(p, device="cuda"), torch.tensor(v, device="cuda")
    depth, path = g4.g4n_locate(ctx, gid, pos, dirs)
    g4.g4n_sync(ctx)
    run = lambda prop: [a.clone() for a in g4.g4n_compute_step(ctx, gid, pos, dirs, depth, path, proposed=prop, mode=mode)]
    bits = lambda b: torch.full((n,), b, dtype=torch.int64, device="cuda").view(torch.float64)
    free = run(None)
    ok = torch.isfinite(free[0])
    assert ok.float().mean() > 0.9
    for b in (0x7ff8000000000000, 0x7ff8000000000000 - (1 << 63), 0x7ff0000000000001, 0x7fffffffffffffff, -1,
              0x7ff0000000000000):
        step, safety, lim = run(bits(b))
        assert torch.equal(step[ok], free[0][ok]) and torch.equal(lim, free[2]), hex(b & (2 ** 64 - 1))
    step, _, lim = run(torch.full((n,), 1e300, dtype=torch.float64, device="cuda"))
    assert torch.equal(step[ok], free[0][ok]) and torch.equal(lim, free[2])
    inside = ok & (free[0] > 0)
    for value in (0.0, -0.0, 5e-324, -5e-324, -1e-300, -3.0, -1e300, -np.inf):
        step, _, lim = run(torch.full((n,), value, dtype=torch.float64, device="cuda"))
        assert torch.all(step[inside] == value) and torch.all(lim[inside] == g4.G4N_LIM_PHYSICS), value
    try:
        g4.g4n_sync(ctx)
    except g4.G4NError:
        pass


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("name", ["mixed", "calorimeter"])
def test_compute_step_from_the_mother_of_the_leaf(env, mode, name):
    """A query may name a volume while its point lies in one of the volume's daughters (a stepping loop that has not yet gone
    down).  The step is the oracle's: zero into a box.  Tolerance: that of the parity tests, 1e-9 mm."""
    import oracle
    from synth.mlp_init import mlp_init
    from gpu_common import mixed_scene
    g4, torch, ctx = env
    g4.g4n_mlp_load(ctx, mlp_init(3))
    sc = mixed_scene(seed=23, n=200, half=200.0) if name == "mixed" else synth.scenes.calorimeter_scene(
        nx=4, ny=4, n_layers=6, voxel=synth.scenes.VoxelSpec())
    og = oracle.Geometry(sc)
    gid = g4.build_scene(ctx, sc)
    rng = np.random.default_rng(24)
    half = np.abs([pl.t for pl in sc.placements[1:] if pl.mother == 0]).max(axis=0) + 10.0
    p, v = rng.uniform(-half, half, (60000, 3)), rng.normal(size=(60000, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    depth, path = og.locate_many(p, v)
    keep = depth > 1
    p, v, depth, path = p[keep], v[keep], depth[keep] - 1, path[keep]
    want, lim_ref, _ = og.compute_step_many(p, v, depth, path)
    T = lambda a, t: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")
    s, _, lim = g4.g4n_compute_step(ctx, gid, T(p.T, torch.float64), T(v.T, torch.float64), T(depth, torch.int32),
                                    T(path.T, torch.int32), mode=mode)
    g4.g4n_sync(ctx)
    s, lim = s.cpu().numpy(), lim.cpu().numpy()
    assert len(p) > 1000 and (want == 0.0).sum() > 100
    assert np.array_equal(lim, lim_ref), (lim != lim_ref).sum()
    assert np.all(np.abs(s - want) <= 1e-9)


@pytest.mark.parametrize("name", ["calorimeter", "barrel", "mixed", "cones", "segments"])
def test_modes_give_the_same_steps(env, name):
    """The three modes choose the crossed surface in their own ways and evaluate it by the same operations: steps and
    limiters agree bit for bit, whichever formulas a query ends in."""
    from synth.mlp_init import mlp_init
    from gpu_common import cones_scene, mixed_scene, segments_scene
    g4, torch, ctx = env
    g4.g4n_mlp_load(ctx, mlp_init(3))
    n = 200000
    if name in ("calorimeter", "barrel"):
        sc = synth.scenes.barrel_scene() if name == "barrel" else synth.scenes.calorimeter_scene(
            voxel=synth.scenes.VoxelSpec(mode="smart"))
        p, v = synth.scenes.query_points(name, n, 34)
    else:
        sc, half = {"mixed": (mixed_scene(seed=23, n=200, half=200.0), 200.0), "cones": (cones_scene(), 480.0),
                    "segments": (segments_scene(), 380.0)}[name]
        rng = np.random.default_rng(35)
        p, v = rng.uniform(-half, half, (3, n)), rng.normal(size=(3, n))
        v /= np.linalg.norm(v, axis=0)
    gid = g4.build_scene(ctx, sc)
    pos, dirs = torch.tensor(p, device="cuda"), torch.tensor(v, device="cuda")
    depth, path = g4.g4n_locate(ctx, gid, pos, dirs)
    prop = torch.tensor(np.random.default_rng(36).exponential(300.0, n), device="cuda")
    got = [[a.cpu().numpy().copy() for a in g4.g4n_compute_step(ctx, gid, pos, dirs, depth, path, proposed=prop, mode=mode)]
           for mode in (0, 1, 2)]
    try:
        g4.g4n_sync(ctx)
    except g4.G4NError:
        pass    # points outside the world
    for mode in (1, 2):
        assert np.array_equal(got[mode][2], got[0][2])
        assert np.array_equal(got[mode][0], got[0][0], equal_nan=True), (got[mode][0] != got[0][0]).sum()


@pytest.mark.parametrize("bad", [float("nan"), -float("nan"), float("inf"), -float("inf"), 1e300, 1e20])
def test_modes_agree_on_points_that_are_no_points(env, bad):
    """compute_step takes a point as it is given: the FP32 mode's answer to a NaN, an infinity or a coordinate beyond any float
    is the FP64 mode's."""
    from gpu_common import mixed_scene
    g4, torch, ctx = env
    gid = g4.build_scene(ctx, mixed_scene(seed=23, n=200, half=200.0))
    rng, n = np.random.default_rng(37), 20000
    p, v = rng.uniform(-150, 150, (3, n)), rng.normal(size=(3, n))
    v /= np.linalg.norm(v, axis=0)
    pos, dirs = torch.tensor(p, device="cuda"), torch.tensor(v, device="cuda")
    depth, path = g4.g4n_locate(ctx, gid, pos, dirs)
    g4.g4n_sync(ctx)
    pos[0, ::2] = bad
    pos[2, ::3] = bad
    got = [[a.cpu().numpy().copy() for a in g4.g4n_compute_step(ctx, gid, pos, dirs, depth, path, mode=mode)] for mode in (0, 1)]
    try:
        g4.g4n_sync(ctx)
    except g4.G4NError:
        pass
    assert np.array_equal(got[0][0], got[1][0], equal_nan=True) and np.array_equal(got[0][2], got[1][2])


@pytest.mark.parametrize("scale", [1e3, 1e6])
@pytest.mark.parametrize("name", ["mixed", "gaps", "segments"])
def test_large_tolerance_scales(env, name, scale):
    """Queries and histories at large tolerances (1e-6 and 1e-3 mm) are the oracle's in every mode, points in surface bands and
    solids a part of the tolerance apart among them."""
    import oracle
    from gpu_common import mixed_scene, random_queries, segments_scene
    from test_portals_host import gap_scene
    g4, torch, _ = env
    sc = {"mixed": lambda: mixed_scene(seed=23, n=150, half=200.0), "gaps": lambda: gap_scene(0.3e-9 * scale),
          "segments": segments_scene}[name]()
    ctx = g4.g4n_create(0)
    oracle.set_scale(scale)
    try:
        g4.g4n_set_tolerance_scale(ctx, scale)
        gid = g4.build_scene(ctx, sc)
        og = oracle.Geometry(sc)
        p, v = random_queries(og, sc, 20000, seed=38, aim_frac=0.5)
        depth, path = og.locate_many(p, v)
        ok = depth > 0
        p, v, depth, path = p[ok], v[ok], depth[ok], path[ok]
        T = lambda a, t: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")
        pos, dirs = T(p.T, torch.float64), T(v.T, torch.float64)
        d, pa = g4.g4n_locate(ctx, gid, pos, dirs)
        assert np.array_equal(d.cpu().numpy(), depth) and np.array_equal(pa.cpu().numpy().T, path)
        want, lim_ref, _ = og.compute_step_many(p, v, depth, path)
        for mode in (0, 1):
            s, _, lim = g4.g4n_compute_step(ctx, gid, pos, dirs, T(depth, torch.int32), T(path.T, torch.int32), mode=mode)
            g4.g4n_sync(ctx)
            assert np.array_equal(lim.cpu().numpy(), lim_ref), (mode, (lim.cpu().numpy() != lim_ref).sum())
            assert np.all(np.abs(s.cpu().numpy() - want) <= 1e-9)
        src = synth.scenes.Source(pos=(15.0, -13.0, 2.0), isotropic=True, e_kind="loguniform", e0=0.05, e1=5.0)
        n = 20000
        ref = og.transport(src, 39, n)["hashes"]
        for mode in (0, 1):
            for schedule, flags in ((0, 0), (1, 0), (1, 1)):
                edep = torch.zeros((100, sc.n_volumes + 2), dtype=torch.float64, device="cuda")
                cnt = torch.zeros(g4.G4N_N_COUNTERS, dtype=torch.int64, device="cuda")
                h = torch.zeros(n, dtype=torch.int64, device="cuda")
                g4.g4n_transport_batch(ctx, g4.make_items([(gid, n, 0, src, 0)]), 39, edep, cnt, h, mode=mode,
                                       schedule=schedule, staged_flags=flags)
                g4.g4n_sync(ctx)
                bad = (h.cpu().numpy().view(np.uint64) != ref).sum()
                assert bad == 0, (mode, schedule, flags, bad)
    finally:
        oracle.set_scale(1.0)
        g4.g4n_destroy(ctx)
