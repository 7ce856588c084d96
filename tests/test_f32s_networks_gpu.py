"""FP32-accurate split decodes (NBTC_FP32 at hidden width 64, NBTC_FP32_TC at
every width) on networks unlike a He initialisation: output biases of the size a
decoder trained on targets in [0, 1] has, channels that are constant, small output
weights, neurons that are pruned.  Every output within the forms' 1e-5 of FP64."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu
TOL_FP32 = 1e-5
SHAPES = [[12, 64, 9], [12, 64, 64, 9], [12, 64, 64, 64, 9], [12, 32, 32, 9], [12, 16, 9]]


@pytest.fixture(scope="module")
def nb():
    require_gpu()
    import paper_2506_06040_gb300 as nb
    return nb


@pytest.fixture(scope="module")
def ctx(nb):
    c = nb.Context(0)
    yield c
    c.close()


def _check(nb, ctx, wl, grid=(150, 40)):
    """FP32 and FP32_TC decodes of a grid against the FP64 oracle."""
    mat = nb.Material.from_synth(wl.material)
    ref = oracle.decode.decode_grid(wl.material, *grid)
    y = nb.decode(ctx, mat, grid=grid)
    z = nb.decode(ctx, mat, nb.FP32_TC, nb.pack_mlp(ctx, mat, nb.FP32_TC), grid=grid)
    ctx.sync()
    for name, t in (("fp32", y), ("fp32_tc", z)):
        err = np.abs(t.cpu().numpy().astype(np.float64) - ref).max(axis=0)
        assert np.all(err <= TOL_FP32), (name, err)  # (NaN fails the comparison)


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("gain,lo,hi", [(1.0, 0.05, 1.0), (0.05, 0.5, 0.5), (1e-3, 0.1, 0.9)])
def test_output_biases(nb, ctx, dims, gain, lo, hi):
    """Biases from a small share of a channel's range to nearly all of it."""
    wl = synth.small_decode_workload(256, dims, seed=700 + len(dims) + dims[1])
    mlp = wl.material.mlp
    mlp.weights[-1] = (mlp.weights[-1] * np.float32(gain)).astype(np.float32)
    mlp.biases[-1] = np.linspace(lo, hi, dims[-1]).astype(np.float32)
    _check(nb, ctx, wl)


@pytest.mark.parametrize("dims", SHAPES)
def test_constant_channels(nb, ctx, dims):
    """Channels without a weight: the bias alone, exactly."""
    wl = synth.small_decode_workload(256, dims, seed=710 + len(dims) + dims[1])
    mlp = wl.material.mlp
    mlp.weights[-1][[0, 4]] = 0.0
    mlp.biases[-1][[0, 4]] = [0.5, 0.0]
    _check(nb, ctx, wl)
    mat = nb.Material.from_synth(wl.material)
    z = nb.decode(ctx, mat, nb.FP32_TC, nb.pack_mlp(ctx, mat, nb.FP32_TC), grid=(64, 4))
    ctx.sync()
    assert bool((z[:, 0] == 0.5).all()) and bool((z[:, 4] == 0.0).all())


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("layer", ["first", "last"])
@pytest.mark.parametrize("share", ["one", "half", "all"])
def test_pruned_neurons(nb, ctx, dims, layer, share):
    """Hidden neurons without an incoming weight or a bias: their activation is 0,
    whatever their outgoing weights, which are ordinary for one and beyond any
    finite scale for the other."""
    wl = synth.small_decode_workload(256, dims, seed=720 + len(dims) + dims[1])
    mlp = wl.material.mlp
    l = 0 if layer == "first" else len(dims) - 3
    n = {"one": 1, "half": dims[1] // 2, "all": dims[1]}[share]
    rows = np.random.default_rng(n).permutation(dims[1])[:n]
    mlp.weights[l][rows] = 0.0
    mlp.biases[l][rows] = 0.0
    mlp.weights[l + 1][:, rows[0]] *= np.float32(1e20)
    _check(nb, ctx, wl)


def _fma_features(material, gw, gh):
    """The 12 features of every texel of a grid as FP32 kernels form them: bytes blended
    down the columns, then along the row, by FMAs, then times RN(1 / 255)."""
    f32 = np.float32
    out = []
    i, j = np.arange(gw * gh) % gw, np.arange(gw * gh) // gw
    for lv in material.levels:
        img = oracle.bc1.decode_level(lv.blocks[0], lv.width, lv.height)[..., :3].astype(np.float64)

        def axis(k, n, size):
            u = oracle.sample.grid_coord(k, n).astype(np.float64)
            t = (u * size + (lv.shift - 0.5)).astype(f32)
            fl = np.floor(t)
            a = fl.astype(int)
            return np.clip(a, 0, size - 1), np.clip(a + 1, 0, size - 1), (t - fl).astype(np.float64)[:, None]

        x0, x1, fx = axis(i, gw, lv.width)
        y0, y1, fy = axis(j, gh, lv.height)
        down = lambda x: (img[y0, x] + fy * (img[y1, x] - img[y0, x])).astype(f32)  # noqa: E731
        left, right = down(x0), down(x1)
        row = (left.astype(np.float64) + fx * (right - left).astype(np.float64)).astype(f32)
        out.append(f32(1.0 / 255.0) * row)
    return np.concatenate(out, axis=1)


def _fma_network(mlp, x):
    """FP32 multiply-adds, inputs in order, bias first."""
    h = x.astype(np.float32)
    for l, (w, b) in enumerate(zip(mlp.weights, mlp.biases)):
        s = np.broadcast_to(b, (len(h), len(b))).astype(np.float32)
        for k in range(w.shape[1]):
            s = (s.astype(np.float64) + h[:, k:k + 1].astype(np.float64) * w[:, k].astype(np.float64)).astype(np.float32)
        h = np.maximum(s, np.float32(0)) if l + 1 < len(mlp.weights) else s
    return h


def _network(kind, mlp, rng):
    ws, bs = mlp.weights, mlp.biases
    if kind == "biases":
        bs[:-1] = [rng.normal(0, 0.1, b.shape) for b in bs[:-1]]
        bs[-1] = rng.uniform(0.1, 0.9, bs[-1].shape)
    elif kind == "positive":
        ws[:] = [np.abs(w) / np.sqrt(w.shape[1]) for w in ws]
    elif kind in ("half", "tenth"):
        q = 0.5 if kind == "half" else 0.1
        ws[:-1] = [w * (rng.random(w.shape) < q) / np.sqrt(q) for w in ws[:-1]]
    elif kind in ("identity", "single"):
        for l, w in enumerate(ws):
            pick = np.arange(len(w)) % w.shape[1] if kind == "identity" else rng.integers(0, w.shape[1], len(w))
            ws[l] = np.zeros_like(w)
            ws[l][np.arange(len(w)), pick] = 1.0 if kind == "identity" else rng.uniform(0.5, 2.0, len(w))
            if kind == "identity":
                bs[l] = np.zeros_like(bs[l])
    elif kind == "dead":  # eight neurons a layer far below their kink
        for b in bs[:-1]:
            b[:8] = -30.0
    mlp.weights, mlp.biases = [w.astype(np.float32) for w in ws], [b.astype(np.float32) for b in bs]


@pytest.mark.parametrize("depth", [1, 2, 3])
@pytest.mark.parametrize("kind,most", [("he", 1.0), ("biases", 1.0), ("positive", 1.0), ("half", 1.0), ("dead", 1.0),
                                       ("identity", 1.0), ("tenth", 2.0), ("single", 2.0)])
def test_error_is_that_of_fp32_multiply_adds(nb, ctx, depth, kind, most):
    """2-norm of the error against FP64 of both forms, over four networks of width 64,
    against that of plain FP32 multiply-adds on the same networks and texels: no larger on
    networks whose rows hold many weights or pass a value on, and at most twice it where a
    row holds one to six weights, whose products FP32 rounds as few times."""
    gw, gh = 256, 48
    ours, plain = np.zeros(2), 0.0
    for seed in range(4):
        wl = synth.small_decode_workload(256, [12] + [64] * depth + [9], seed=730 + 10 * depth + seed)
        _network(kind, wl.material.mlp, np.random.default_rng(seed))
        mat = nb.Material.from_synth(wl.material)
        y = nb.decode(ctx, mat, grid=(gw, gh))
        z = nb.decode(ctx, mat, nb.FP32_TC, nb.pack_mlp(ctx, mat, nb.FP32_TC), grid=(gw, gh))
        ctx.sync()
        ref = oracle.decode.decode_grid(wl.material, gw, gh)
        scale = np.linalg.norm(ref)
        plain += (np.linalg.norm(_fma_network(wl.material.mlp, _fma_features(wl.material, gw, gh)) - ref) / scale) ** 2
        ours += [(np.linalg.norm(t.cpu().numpy().astype(np.float64) - ref) / scale) ** 2 for t in (y, z)]
    ratio = np.sqrt(ours / plain)
    print(f"{kind} {depth}: plain FP32 {np.sqrt(plain / 4):.2e}, ratio {ratio}")
    assert np.all(ratio <= most), ratio
