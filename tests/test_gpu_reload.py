"""Particles loaded into a handle that holds others: sizes at which the buffers' block is kept
(as many, slightly fewer) and at which it is allocated anew (far fewer, more), against a
fresh handle, bit by bit; and outputs that kernels write in place against staged ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params, lattice_bed  # noqa: E402


def handle(form):
    return sedi.Sedi(dict(default_params(hi=(8e-3, 8e-3, 16e-3), ncell=(8, 7, 9), wall_hi=(0, 0, 0)),
                          precision_form=form))


def load(h, n, seed):
    g = np.random.default_rng(seed)
    x = lattice_bed(n, 8e-3, 0.5e-3, seed, jitter=2e-4, spacing=1.0)
    h.set_particles(x, 1e-2 * g.normal(size=(n, 3)), g.normal(size=(n, 3)), np.full(n, 0.5e-3), np.full(n, 2500.0))
    h.set_eps(np.full(h.C, 0.1))  # the drag's solid fraction stays with the mesh
    f = h.compute_forces()
    off, ids = h.neighbors()
    eps, us, fd = h.average()
    h.step(3)
    return [f[k] for k in sorted(f)] + [off, ids, eps, us, fd, h.get_particles()[0]]


@pytest.mark.parametrize("form", ["split", "fp64"])
def test_reload_equals_a_fresh_handle(form):
    h = handle(form)
    for k, n in enumerate((1500, 1500, 1497, 1, 33, 2100)):
        for a, b in zip(load(h, n, k), load(handle(form), n, k)):
            np.testing.assert_array_equal(a, b)


def test_outputs_in_place_equal_staged_ones():
    h = handle("split")
    load(h, 700, 3)
    C = h.C
    host = h.average()
    dev = [torch.full(s, 7.0, dtype=torch.float64, device="cuda") for s in ((C,), (C, 3), (C, 3))]
    h.average(*dev)
    pos = torch.full((700, 3), 7.0, dtype=torch.float64, device="cuda")
    h.get_positions(pos)
    for a, b in zip(host + (h.get_positions(np.zeros((700, 3))),), dev + [pos]):
        np.testing.assert_array_equal(a, b.cpu().numpy())
    h.average(dev[0])  # one output alone
    np.testing.assert_array_equal(h.average()[0], dev[0].cpu().numpy())
