"""A checkpoint loaded into a handle that already holds as many particles, whose buffers are
kept, and that has steps in flight, against the same checkpoint in a fresh handle: the
stored state, the fluid fields and what follows from them, bit by bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import small_case  # noqa: E402


def state(h):
    ij, xi = h.contacts()
    out = [ij, xi, h.wall_springs(), *h.neighbors(), *h.get_particles()]
    h.step(10)
    return out + [*h.get_particles(), *h.average()]


@pytest.mark.parametrize("form", ["split", "plain", "fp64"])
def test_checkpoint_into_a_used_handle(form, tmp_path):
    prm, parts = small_case(parity_addon=True)
    prm = dict(prm, precision_form=form)
    args = [parts[k] for k in ("x", "v", "w", "d", "rho")]
    U = np.random.default_rng(3).normal(0.0, 0.05, (int(np.prod(prm["ncell"])), 3))
    src = sedi.Sedi(prm)
    src.set_particles(*args)
    src.set_fluid(U=U)
    src.step(15)
    path = tmp_path / "state"
    src.save_state(path)
    fresh = sedi.Sedi(prm)
    fresh.load_state(path)
    fresh.n = len(parts["d"])
    want = state(fresh)
    used = sedi.Sedi(prm)
    for k in range(8):
        used.set_particles(*args)
        used.set_fluid(U=2.0 * U)
        used.step(10 * k)
        used.load_state(path)
        used.n = len(parts["d"])
        for a, b in zip(state(used), want):
            if form == "plain":  # its averaging adds in an order of its own each time
                np.testing.assert_allclose(a, b, rtol=1e-3, atol=1e-4 * max(np.abs(b).max(), 1e-300))
            else:
                np.testing.assert_array_equal(a, b)
