"""The learned candidate proposal on the GPU: inference and gradients against the
FP64 reference network, training on samples logged by the plain navigator, identical
transport results in learned mode, and what the trained network saves."""
import math

import numpy as np
import pytest

import oracle
from oracle import mlp as omlp
import synth
from synth.mlp_init import mlp_init
from gpu_common import mixed_scene

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


def random_data(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.uniform(-1, 1, (n, 9)).astype(np.float32)
    nc = rng.integers(2, 33, n).astype(np.int32)
    X[:, 7] = nc / 32.0
    X[:, 8] = 1.0
    y = np.array([rng.integers(0, k) for k in nc], dtype=np.int32)
    return X, y, nc


def params(seed):
    return (mlp_init(seed) + np.random.default_rng(seed).normal(0, 0.05, omlp.N_PARAMS)).astype(np.float32)


def test_predict_matches_reference(env):
    g4, torch, ctx = env
    p = params(5)
    g4.g4n_mlp_load(ctx, p)
    assert np.array_equal(g4.g4n_mlp_get(ctx), p)
    X, _, nc = random_data(1001, 6)   # ragged: not a multiple of the 32-row warp tile
    logits = g4.g4n_mlp_predict(ctx, torch.tensor(X, device="cuda")).cpu().numpy()
    ref, _ = omlp.forward(p, X, emulate_bf16=True)
    assert np.all(np.abs(logits - ref) <= 0.03 + 0.02 * np.abs(ref)), np.max(np.abs(logits - ref))
    top2 = np.sort(ref, axis=1)[:, -2:]
    clear = top2[:, 1] - top2[:, 0] > 0.1
    assert np.all(np.argmax(logits, axis=1)[clear] == np.argmax(ref, axis=1)[clear])


@pytest.mark.parametrize("precision,rtol", [(1, 1e-5), (0, 2e-2)])
def test_gradients_match_reference(env, precision, rtol):
    g4, torch, ctx = env
    p = params(7)
    g4.g4n_mlp_load(ctx, p)
    X, y, nc = random_data(512, 8)
    T = lambda a: torch.tensor(a, device="cuda")
    loss, g = g4.g4n_mlp_grad(ctx, T(X), T(y), T(nc), precision=precision)
    ref_loss, ref_g = omlp.loss_and_grad(p.astype(np.float64), X.astype(np.float64), y, nc)
    assert abs(loss - ref_loss) <= max(rtol, 1e-6) * abs(ref_loss)
    for got, want in zip(omlp.unpack(g), omlp.unpack(ref_g)):
        assert np.linalg.norm(got - want) <= rtol * np.linalg.norm(want) + 1e-12


def _items(g4, gid, n, src, tid0=0):
    return g4.make_items([(gid, n, tid0, src, 0)])


def test_logging_and_training(env):
    g4, torch, ctx = env
    sc = mixed_scene(seed=9, n=400, half=300.0)
    gid = g4.build_scene(ctx, sc)
    src = synth.scenes.Source(pos=(0.0, 0.0, 0.0), isotropic=True, e_kind="loguniform", e0=0.05, e1=5.0)
    feat, label, ncand = g4.g4n_mlp_log(ctx, _items(g4, gid, 200000, src), 11, 400000, sc.n_volumes + 2)
    n = feat.shape[0]
    assert n > 10000
    lab, nc, F = label.cpu().numpy(), ncand.cpu().numpy(), feat.cpu().numpy()
    assert np.all((nc >= 2) & (nc <= 32) & (lab >= 0) & (lab < nc))
    assert np.all(np.abs(F[:, :3]) <= 2.0) and np.allclose(np.linalg.norm(F[:, 3:6], axis=1), 1.0, atol=1e-6)
    assert np.allclose(F[:, 7], nc / 32.0) and np.all(F[:, 8] == 1.0)
    g4.g4n_mlp_load(ctx, mlp_init(12))
    losses = g4.g4n_mlp_train(ctx, feat, label, ncand, epochs=4, batch=1024, lr=2e-3, seed=3)
    assert losses[-1] < losses[0] < math.log(32)
    pred = g4.g4n_mlp_predict(ctx, feat).cpu().numpy()
    pred = np.where(np.arange(32)[None, :] < nc[:, None], pred, -np.inf).argmax(axis=1)
    acc = (pred == lab).mean()
    base = max(np.mean(lab == 0), np.mean(lab == np.bincount(lab).argmax()))
    # better than always proposing the most common slot: the error rate drops by a fifth at least
    assert (1.0 - acc) < 0.8 * (1.0 - base), (acc, base)


@pytest.mark.parametrize("name", ["mixed", "barrel"])
def test_learned_transport_identical(env, name):
    g4, torch, ctx = env
    sc = mixed_scene(seed=10, n=300, half=300.0) if name == "mixed" else synth.scenes.barrel_scene()
    src = (synth.scenes.Source(pos=(5.0, -3.0, 2.0), isotropic=True, e_kind="loguniform", e0=0.05, e1=5.0)
           if name == "mixed" else synth.scenes.barrel_source())
    gid = g4.build_scene(ctx, sc)
    g4.g4n_mlp_load(ctx, mlp_init(21))
    n, seed = 20000, 4321
    og = oracle.Geometry(sc)
    r = og.transport(src, seed, n)
    out = {}
    for mode in (0, 1, 2):
        edep = torch.zeros((100, sc.n_volumes + 2), dtype=torch.float64, device="cuda")
        cnt = torch.zeros(32, dtype=torch.int64, device="cuda")
        h = torch.zeros(n, dtype=torch.int64, device="cuda")
        g4.g4n_transport_batch(ctx, _items(g4, gid, n, src), seed, edep, cnt, h, mode=mode, diagnostics=True)
        g4.g4n_sync(ctx)
        out[mode] = (h.cpu().numpy().view(np.uint64), g4.counters_dict(cnt), edep.cpu().numpy().sum(axis=0))
        assert np.array_equal(out[mode][0], r["hashes"]), mode
        for k, nm in enumerate(oracle.COUNTER_NAMES[:10]):
            assert out[mode][1][nm] == int(r["counters"][k]), (mode, nm)
    assert out[2][1]["proposals"] > 0


def test_trained_proposal_saves_exact_evaluations(env):
    """What the trained network gains, at identical histories, on random worlds (voxel lists in id order,
    the first-hit daughter already first in most nodes): the plain navigator evaluates every listed
    candidate in FP64; the learned mode evaluates the proposal first and prunes the rest by the rigorous
    FP32 bounds, as many evaluations as the FP32 bounds alone or fewer."""
    g4, torch, ctx = env
    sc = mixed_scene(seed=13, n=1500, half=400.0)
    gid = g4.build_scene(ctx, sc)
    src = synth.scenes.Source(pos=(0.0, 0.0, 0.0), isotropic=True, e_kind="loguniform", e0=0.05, e1=5.0)
    feat, label, ncand = g4.g4n_mlp_log(ctx, _items(g4, gid, 300000, src, tid0=10_000_000), 5, 1_000_000,
                                        sc.n_volumes + 2)
    g4.g4n_mlp_load(ctx, mlp_init(14))
    g4.g4n_mlp_train(ctx, feat, label, ncand, epochs=6, batch=2048, lr=2e-3, seed=4)
    res = _evaluations(env, gid, sc, src, 200000, 99)
    plain_evals = sum(res[0][1][k] for k in ("cand_box", "cand_tube", "cand_orb"))
    fp32_evals = res[1][1]["rechecks"]
    learned_evals = res[2][1]["rechecks"]
    print(f"FP64 candidate evaluations: plain {plain_evals}, fp32 bounds {fp32_evals}, learned {learned_evals}, "
          f"proposals {res[2][1]['proposals']}, pruned {res[2][1]['pruned']}")
    assert learned_evals <= fp32_evals
    assert learned_evals < 0.25 * plain_evals


def _evaluations(env, gid, sc, src, n, seed):
    g4, torch, ctx = env
    res = {}
    for mode in (0, 1, 2):
        edep = torch.zeros((100, sc.n_volumes + 2), dtype=torch.float64, device="cuda")
        cnt = torch.zeros(32, dtype=torch.int64, device="cuda")
        h = torch.zeros(n, dtype=torch.int64, device="cuda")
        g4.g4n_transport_batch(ctx, _items(g4, gid, n, src), seed, edep, cnt, h, mode=mode, diagnostics=True)
        g4.g4n_sync(ctx)
        res[mode] = (h.cpu().numpy(), g4.counters_dict(cnt))
    assert np.array_equal(res[0][0], res[2][0]) and np.array_equal(res[1][0], res[2][0])
    return res


def test_trained_proposal_gains_where_list_order_misleads(env):
    """The gain of the trained network over the method without it (the FP32-bounded navigator), at
    identical histories and against the oracle: in a stack of plates numbered from the far end, the
    candidate list puts the plates an upward ray reaches last first, so the bounds alone evaluate every
    plate ahead of the ray in FP64, farthest first; the trained proposal names the next plate, whose
    exact distance then prunes the rest."""
    g4, torch, ctx = env
    sc = synth.scenes.reversed_stack_scene()
    src = synth.scenes.reversed_stack_source()
    gid = g4.build_scene(ctx, sc)
    feat, label, ncand = g4.g4n_mlp_log(ctx, _items(g4, gid, 100000, src, tid0=20_000_000), 7, 1_000_000,
                                        sc.n_volumes + 2)
    assert feat.shape[0] > 100000
    g4.g4n_mlp_load(ctx, mlp_init(15))
    losses = g4.g4n_mlp_train(ctx, feat, label, ncand, epochs=4, batch=2048, lr=2e-3, seed=6)
    n, seed = 50000, 77
    res = _evaluations(env, gid, sc, src, n, seed)
    r = oracle.Geometry(sc).transport(src, seed, n)
    assert np.array_equal(res[2][0].view(np.uint64), r["hashes"])
    fp32_evals = res[1][1]["rechecks"]
    learned_evals = res[2][1]["rechecks"]
    print(f"losses {losses.tolist()}; FP64 candidate evaluations: fp32 bounds {fp32_evals}, learned {learned_evals}, "
          f"proposals {res[2][1]['proposals']}, pruned {res[2][1]['pruned']}, steps {res[2][1]['steps']}")
    assert learned_evals < 0.5 * fp32_evals


def test_trained_learned_barrel_full_size_sampled(env):
    """The learned mode with a trained network on the barrel at full size (10^7 tracks): identical
    histories to the plain FP64 navigator, and 300 sampled histories replayed one by one by the oracle."""
    g4, torch, ctx = env
    sc = synth.scenes.barrel_scene()
    src = synth.scenes.barrel_source()
    gid = g4.build_scene(ctx, sc)
    feat, label, ncand = g4.g4n_mlp_log(ctx, _items(g4, gid, 500000, src, tid0=50_000_000), 3, 2_000_000,
                                        sc.n_volumes + 2)
    g4.g4n_mlp_load(ctx, mlp_init(41))
    losses = g4.g4n_mlp_train(ctx, feat, label, ncand, epochs=2, batch=4096, lr=2e-3, seed=5)
    assert losses[-1] < losses[0]
    del feat, label, ncand
    n, seed = 10_000_000, synth.scenes.CONFIG_SEEDS[4][1]
    hashes = {}
    # the plain navigator, the learned mode with its counters (persistent kernel), the learned mode staged
    for mode, diag, sched in ((0, False, 0), (2, True, 0), (2, False, 1)):
        edep = torch.zeros((100, sc.n_volumes + 2), dtype=torch.float64, device="cuda")
        cnt = torch.zeros(32, dtype=torch.int64, device="cuda")
        h = torch.zeros(n, dtype=torch.int64, device="cuda")
        g4.g4n_transport_batch(ctx, _items(g4, gid, n, src), seed, edep, cnt, h, mode=mode, diagnostics=diag,
                               schedule=sched)
        g4.g4n_sync(ctx)
        hashes[mode, sched] = h.cpu().numpy().view(np.uint64)
        c = g4.counters_dict(cnt)
        assert c["tracks"] == n and c["steps"] == c["geom_steps"] + c["phys_steps"]
        if diag:
            assert c["proposals"] > 0
        del edep, cnt, h
    for key in ((2, 0), (2, 1)):
        bad = np.nonzero(hashes[0, 0] != hashes[key])[0]
        assert bad.size == 0, f"{bad.size} histories differ between the plain navigator and {key}"
    og = oracle.Geometry(sc)
    for i in np.unique(np.random.default_rng(8).integers(0, n, 300)):
        r = og.transport(src, seed, 1, tid0=int(i), threads=1)
        assert hashes[2, 1][i] == r["hashes"][0], i


@pytest.mark.parametrize("n", [16, 32, 48, 768, 784, 4864, 4880, 9760])
def test_bf16_gradients_at_tile_edges(env, n):
    """Small batches of the plain kernels, the first and a ragged one of the persistent kernel, one tile per SM of a 152-SM GPU, one row block more, two tiles on
    some blocks and a ragged one.  Tolerance: that of the BF16 gradients above (8 significant bits, 2e-2 in norm)."""
    g4, torch, ctx = env
    p = params(27)
    g4.g4n_mlp_load(ctx, p)
    X, y, nc = random_data(n, 28)
    T = lambda a: torch.tensor(a, device="cuda")
    loss, g = g4.g4n_mlp_grad(ctx, T(X), T(y), T(nc), precision=0)
    ref_loss, ref_g = omlp.loss_and_grad(p.astype(np.float64), X.astype(np.float64), y, nc)
    assert abs(loss - ref_loss) <= 2e-2 * abs(ref_loss)
    for got, want in zip(omlp.unpack(g), omlp.unpack(ref_g)):
        assert np.linalg.norm(got - want) <= 2e-2 * np.linalg.norm(want) + 1e-12
    again = g4.g4n_mlp_grad(ctx, T(X), T(y), T(nc), precision=0)
    assert again[0] == loss and np.array_equal(again[1], g)   # the summation order is fixed


@pytest.mark.parametrize("batch", [16, 48, 768, 4880])
def test_training_step_matches_its_gradient(env, batch):
    """One minibatch of an epoch: its loss is that of the permuted samples, and the update is Adam's first step on
    their gradient (the same kernel's, over the same rows in the same order).  Tolerance: the update in FP32 from the
    same gradient, a few roundings of relative 2^-24 in the step and one in the parameter."""
    g4, torch, ctx = env
    p, n, seed, lr = params(31), batch + 7, 9, np.float32(2e-3)
    X, y, nc = random_data(n, 32)
    wrap = (1 << 64) - 1
    h = (seed * 0x9E3779B97F4A7C15 + 1) & wrap
    h ^= h >> 31
    h = (h * 0xBF58476D1CE4E5B9) & wrap
    h ^= h >> 27
    stride = (h % n) | 1
    while math.gcd(stride, n) != 1:
        stride += 2
    rows = np.array([(r * stride + (h >> 17) % n) % n for r in range(batch)])
    T = lambda a: torch.tensor(a, device="cuda")
    g4.g4n_mlp_load(ctx, p)
    loss, g = g4.g4n_mlp_grad(ctx, T(X[rows]), T(y[rows]), T(nc[rows]))
    losses = g4.g4n_mlp_train(ctx, T(X), T(y), T(nc), epochs=1, batch=batch, lr=float(lr), seed=seed)
    assert abs(losses[0] - loss) <= 1e-6 * loss
    f = np.float32
    m, v = (f(1) - f(0.9)) * g, (f(1) - f(0.999)) * g * g
    c1, c2 = f(1) / (f(1) - f(0.9)), f(1) / (f(1) - f(0.999))
    step = lr * (m * c1) / (np.sqrt(v * c2) + f(1e-8))
    got = g4.g4n_mlp_get(ctx)
    assert np.all(np.abs(got - (p - step)) <= 2.0 ** -23 * np.abs(p) + 1e-6 * np.abs(step) + 1e-12)


@pytest.mark.parametrize("scale", [0.1, 1.0, 10.0])
@pytest.mark.parametrize("n", [1, 16, 17, 32, 33, 129])
def test_predict_rows_and_activation_range(env, n, scale):
    """Row counts around the 16-row halves and the 32-row tiles; weights that keep the hidden layers' inputs near zero, around
    one, and far out in GELU's tails.  A row does not depend on its batch, and lies within one BF16 unit per hidden value
    (2^-8, carried through the layers; GELU's slope is below 1.13) plus the FP32 sums' rounding of the emulated pass."""
    g4, torch, ctx = env
    p = (params(11) * scale).astype(np.float32)
    g4.g4n_mlp_load(ctx, p)
    X, _, _ = random_data(160, 12)
    full = g4.g4n_mlp_predict(ctx, torch.tensor(X, device="cuda")).cpu().numpy()
    part = g4.g4n_mlp_predict(ctx, torch.tensor(X[:n], device="cuda")).cpu().numpy()
    assert np.array_equal(part, full[:n])
    ref, _ = omlp.forward(p, X, emulate_bf16=True)
    b16 = lambda a: torch.tensor(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()
    W1, b1, W2, b2, W3, b3 = [np.asarray(a, dtype=np.float64) for a in omlp.unpack(p)]
    W1, W2, W3 = b16(W1), b16(W2), b16(W3)
    h1 = b16(omlp.gelu(b16(X) @ W1 + b1))
    h2 = b16(omlp.gelu(h1 @ W2 + b2))
    u, f = 2.0 ** -8, 128 * 2.0 ** -23
    e1 = u * np.abs(h1) + 1.13 * f * (np.abs(b16(X)) @ np.abs(W1) + np.abs(b1)) + 1e-6
    e2 = u * np.abs(h2) + 1.13 * (e1 @ np.abs(W2) + f * (np.abs(h1) @ np.abs(W2) + np.abs(b2))) + 1e-6
    e3 = e2 @ np.abs(W3) + f * (np.abs(h2) @ np.abs(W3) + np.abs(b3)) + 1e-6
    assert np.all(np.abs(full - ref) <= e3)


def gradient_chunk(n):
    """Rows of a partial weight gradient: 256 or a little more, a multiple of 16, at most 256 partials."""
    split = max(1, min(256, n // 256))
    return -(-(-(-n // split)) // 16) * 16


@pytest.mark.parametrize("n", [1024, 1088, 2048, 2176, 4096])
def test_gradient_is_the_ascending_sum_of_its_chunks(env, n):
    """Training's rounding of the weights to BF16 makes another grouping of a gradient's sums another training: a weight
    gradient over many rows is, bit for bit, the FP32 sum of the chunks' gradients in ascending order.  The number of
    chunks is a power of two, so that a chunk's own gradient (a mean over its rows) scales exactly."""
    g4, torch, ctx = env
    g4.g4n_mlp_load(ctx, params(41))
    X, y, nc = random_data(n, 42)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    chunk = gradient_chunk(n)
    chunks = n // chunk
    assert chunk * chunks == n and chunks & (chunks - 1) == 0 and chunk < 512
    want = np.zeros(omlp.N_PARAMS, dtype=np.float32)
    for z in range(chunks):
        rows = slice(z * chunk, (z + 1) * chunk)
        want += g4.g4n_mlp_grad(ctx, T(X[rows]), T(y[rows]), T(nc[rows]))[1] * np.float32(1.0 / chunks)
    got = omlp.unpack(g4.g4n_mlp_grad(ctx, T(X), T(y), T(nc))[1])
    for name, k in (("W1", 0), ("W2", 2), ("W3", 4)):
        assert np.array_equal(got[k], omlp.unpack(want)[k]), name


def test_bias_gradient_is_the_column_sum(env):
    """The order of a bias gradient's sum: 256 partial sums of every 256th row, a butterfly over 32 of them, the eight
    results in ascending order; bit for bit.  A row's own term comes from a batch of it and rows without a gradient (one
    candidate: its probability is one)."""
    g4, torch, ctx = env
    n = 1024
    g4.g4n_mlp_load(ctx, params(43))
    X, y, nc = random_data(n, 44)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    bias = lambda g: np.concatenate([omlp.unpack(g)[k].ravel() for k in (1, 3, 5)])
    feat, label, ncand = T(X), T(y), T(nc)
    F, L, N = feat[:16].clone(), torch.zeros(16, dtype=torch.int32, device="cuda"), torch.ones(16, dtype=torch.int32, device="cuda")
    rows = np.empty((n, 160), dtype=np.float32)
    for r in range(n):
        F[0], L[0], N[0] = feat[r], label[r], ncand[r]
        rows[r] = bias(g4.g4n_mlp_grad(ctx, F, L, N)[1]) * np.float32(16.0 / n)
    acc = np.zeros((256, 160), dtype=np.float32)
    for j in range(n // 256):
        acc += rows[256 * j:256 * (j + 1)]
    acc = acc.reshape(8, 32, 160)
    for o in (16, 8, 4, 2, 1):
        acc = acc + acc[:, np.arange(32) ^ o]
    want = np.zeros(160, dtype=np.float32)
    for w in range(8):
        want += acc[w, 0]
    assert np.array_equal(bias(g4.g4n_mlp_grad(ctx, feat, label, ncand)[1]), want)


def test_loss_of_many_rows_is_summed_in_fp64(env):
    """A row's loss is an FP32 value, their sum is not: the loss over 2^17 rows is that of its parts of 512 rows, whose sums the
    plain kernels take row by row in FP64.  Tolerance: a rounding of 2^-53 per row."""
    g4, torch, ctx = env
    n = 1 << 17
    g4.g4n_mlp_load(ctx, params(45))
    X, y, nc = random_data(n, 46)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    feat, label, ncand = T(X), T(y), T(nc)
    parts = [g4.g4n_mlp_grad(ctx, feat[k:k + 512], label[k:k + 512], ncand[k:k + 512])[0] for k in range(0, n, 512)]
    want = math.fsum(parts) / len(parts)
    loss, _ = g4.g4n_mlp_grad(ctx, feat, label, ncand)
    assert abs(loss - want) <= n * 2.0 ** -53 * want, (loss, want)


def test_first_training_on_a_side_stream(env):
    """The buffers of a context's first training are made ready on the training's own stream: with work queued on the default
    stream, which a side stream does not wait for, its weights are those of a training on an idle device."""
    g4, torch, _ = env
    X, y, nc = random_data(4096, 48)
    data = [torch.tensor(a, device="cuda") for a in (X, y, nc)]
    got = []
    for busy in (False, True):
        ctx = g4.g4n_create(0)
        try:
            g4.g4n_mlp_load(ctx, params(47))
            torch.cuda.synchronize()
            side = torch.cuda.Stream()
            if busy:
                torch.cuda._sleep(200_000_000)   # cycles: a tenth of a second of the default stream
            g4.g4n_mlp_train(ctx, *data, epochs=2, batch=2048, lr=2e-3, seed=3, stream=side)
            torch.cuda.synchronize()
            got.append(g4.g4n_mlp_get(ctx))
        finally:
            g4.g4n_destroy(ctx)
    assert np.array_equal(got[0], got[1])
