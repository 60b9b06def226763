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
