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
