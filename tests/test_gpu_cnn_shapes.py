"""The network on meshes whose sizes its kernels do not divide: odd cell counts (the parts
of the work space after an odd number of 8-byte words), axes of one cell, rows shorter
than a warp, and every mix of wrapped and zero-padded axes, against the FP64 reference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as orc  # noqa: E402
from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params  # noqa: E402



def params(seed):
    rng = np.random.default_rng(seed)
    p = []
    for ci, co in ((4, 32), (32, 32), (32, 4)):
        p += [rng.normal(0, np.sqrt(2.0 / (27 * ci)), co * ci * 27), rng.normal(0, 0.05, co)]
    return np.concatenate(p)


@pytest.mark.parametrize("ncell,periodic", [
    ((5, 7, 9), (1, 1, 0)), ((1, 1, 1), (1, 1, 0)), ((1, 3, 33), (0, 0, 0)), ((33, 1, 3), (1, 0, 1)),
    ((17, 9, 5), (0, 1, 1)), ((16, 8, 4), (1, 1, 1)), ((31, 13, 11), (1, 1, 0)), ((64, 2, 3), (0, 0, 1))])
def test_forward_and_gradient_on_ragged_meshes(ncell, periodic):
    """bfloat16 storage at the same points on both sides: what is left is FP32 against FP64
    accumulation, 27 x 32 products an output (~1e-6), and activations that it makes round
    to the other bfloat16 neighbour (2^-8 of one activation, a few of thousands)."""
    hi = tuple(1e-3 * n for n in ncell)
    g = sedi.Sedi(default_params(hi=hi, ncell=ncell, periodic=periodic, wall_lo=(0, 0, 0), wall_hi=(0, 0, 0)))
    p = params(11)
    g.cnn_set_params(p)
    C = int(np.prod(ncell))
    rng = np.random.default_rng(12)
    x, t = rng.normal(0, 1, (4, C)), rng.normal(0, 1, (4, C))
    y = g.cnn_forward(x)
    ref = orc.cnn_forward(p, x, ncell, periodic, round_bf16=True)
    assert np.abs(y - ref).max() <= 2e-2 * np.abs(ref).max()
    assert np.abs(y - ref).mean() <= 1e-3 * np.abs(ref).max()
    loss, grad = g.cnn_loss_grad(x, t)
    loss_ref, grad_ref = orc.cnn_loss_grad(p, x, t, ncell, periodic)
    assert abs(loss - loss_ref) <= 2e-2 * loss_ref
    assert np.linalg.norm(grad - grad_ref) < 5e-2 * np.linalg.norm(grad_ref)


@pytest.mark.parametrize("ncell,periodic", [
    ((8, 8, 4), (1, 1, 0)), ((9, 8, 5), (0, 1, 1)), ((7, 9, 3), (1, 0, 1)), ((16, 4, 8), (0, 0, 0)),
    ((1, 1, 1), (1, 1, 1)), ((2, 33, 9), (1, 1, 1)), ((41, 37, 30), (1, 1, 0))])
def test_exact_sums_at_tile_edges(ncell, periodic):
    """Fields of -1, 0, 1 and sparse weights of the same: every activation is a whole number
    below 256, a bfloat16 word, so the output is exact, and the gradients differ from the FP64
    ones by their FP32 sums alone: a random walk over 27 x 32 products and the voxels,
    sqrt(5e4) 2^-25 = 7e-6 at the largest mesh if nothing were summed in parts."""
    hi = tuple(1e-3 * n for n in ncell)
    g = sedi.Sedi(default_params(hi=hi, ncell=ncell, periodic=periodic, wall_lo=(0, 0, 0), wall_hi=(0, 0, 0)))
    rng = np.random.default_rng(31)
    p = np.concatenate([rng.integers(-1, 2, n) * (rng.random(n) < q) for n, q in (
        (3456, .2), (32, 1), (27648, .04), (32, 1), (3456, .2), (4, 1))]).astype(np.float64)
    g.cnn_set_params(p)
    C = int(np.prod(ncell))
    x, t = rng.integers(-1, 2, (4, C)).astype(float), rng.integers(-9, 10, (4, C)).astype(float)
    np.testing.assert_array_equal(g.cnn_forward(x), orc.cnn_forward(p, x, ncell, periodic, round_bf16=True))
    loss, grad = g.cnn_loss_grad(x, t)
    loss_ref, grad_ref = orc.cnn_loss_grad(p, x, t, ncell, periodic)
    assert abs(loss - loss_ref) <= 1e-12 * loss_ref
    assert np.linalg.norm(grad - grad_ref) <= 7e-6 * np.linalg.norm(grad_ref)
