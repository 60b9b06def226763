"""FP64 ensembles: the averaging of every bed to the bits that it has alone, for few beds and for
many, small and larger ones (the smoother streams small meshes in one launch for all and gives
larger ones the chip in turn); and what many small beds cost."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params  # noqa: E402


def beds(meshes):
    """A jittered lattice of spheres in each bed, moving."""
    out = []
    for b, nc in enumerate(meshes):
        g = np.random.default_rng(100 + b)
        hi = 1e-3 * np.array(nc)
        k = np.maximum(np.minimum(nc, 6), 1)
        x = (np.stack(np.meshgrid(*[(np.arange(n) + 0.5) / n for n in k], indexing="ij"), -1).reshape(-1, 3)) * hi
        x += g.uniform(-1e-4, 1e-4, x.shape)
        n = len(x)
        out.append((nc, hi, (x, g.normal(0.0, 0.05, (n, 3)), np.zeros((n, 3)), np.full(n, 0.5e-3), np.full(n, 2500.0))))
    return out


def ensemble(bs):
    e = sedi.Sedi(dict(default_params(), n_beds=len(bs), precision_form="fp64"))
    for b, (nc, hi, p) in enumerate(bs):
        e.set_bed(b, (0.0, 0.0, 0.0), hi, nc)
        e.set_particles(*p, bed=b)
    return e


@pytest.mark.parametrize("meshes", [
    [(8, 8, 8), (5, 7, 9)],                                      # few and small: the chip in turn
    [(8, 8, 8), (7, 6, 9), (12, 11, 10)] * 8,                    # many and small: one launch
    [(40, 41, 39), (8, 8, 8), (36, 44, 48), (9, 8, 7)],          # large ones on chip, small ones too
    [(40, 41, 39)] + [(16, 15, 14), (9, 8, 7)] * 10,             # large on chip, small streamed
])
def test_beds_have_the_bits_they_have_alone(meshes):
    bs = beds(meshes)
    e = ensemble(bs)
    e.average_inplace()
    for b, (nc, hi, p) in enumerate(bs):
        if b > 6 and b < len(bs) - 2:
            continue
        g = sedi.Sedi(dict(default_params(), lo=(0.0, 0.0, 0.0), hi=tuple(hi), ncell=nc, precision_form="fp64"))
        g.set_particles(*p)
        for one, many in zip(g.average(), e.average(bed=b)):
            np.testing.assert_array_equal(one, many)
        g.close()


def test_many_small_beds_share_the_chip():
    """64 beds of 8^3 cells, 128 units for 152 SMs, against 2 beds: one streaming launch takes
    about 4 times what two on chip do; one after the other on chip they took 31 times."""
    def timed(n):
        e = ensemble(beds([(8, 8, 8)] * n))
        t = []
        for _ in range(6):
            t0 = time.perf_counter()
            e.average_inplace()
            t.append(time.perf_counter() - t0)
        return float(np.median(t))

    t2, t64 = timed(2), timed(64)
    assert t64 <= 10.0 * t2, (t2, t64)


def test_beds_share_the_room_for_tagged_words():
    """64 beds of 8^3 cells hold about 0.5 MB each; room of its own made it 4.5 MB a bed."""
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    e = ensemble(beds([(8, 8, 8)] * 64))
    e.average_inplace()
    used = free - torch.cuda.mem_get_info()[0]
    e.close()
    assert used <= 64 * 2e6, used


@pytest.mark.parametrize("form", ["fp64", "split", "plain"])
def test_a_bed_smooths_as_a_handle_does(form):
    """Fields of a caller through a bed, whose room for tagged words is the ensemble's and grows
    with later beds, and through a handle."""
    prm = dict(default_params(), precision_form=form)
    e = sedi.Sedi(dict(prm, n_beds=3))
    meshes = [(8, 9, 7), (19, 15, 31), (53, 51, 49)]
    for b, nc in enumerate(meshes):
        hi = tuple(1e-3 * n for n in nc)
        e.set_bed(b, (0.0, 0.0, 0.0), hi, nc)
        for k in range(b + 1):
            phi = np.random.default_rng(k).random((3, int(np.prod(meshes[k]))))
            g = sedi.Sedi(dict(prm, hi=tuple(1e-3 * n for n in meshes[k]), ncell=meshes[k]))
            out, it = e.smooth(phi, bed=k)
            ref, ir = g.smooth(phi)
            np.testing.assert_array_equal(out, ref)
            np.testing.assert_array_equal(it, ir)
            g.close()
