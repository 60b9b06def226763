"""Outputs into host arrays: the forces of few particles (one copy for the four arrays) and of
more against device outputs, and large arrays whose pages the process has not touched."""
import ctypes
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params, lattice_bed  # noqa: E402


def handle(n):
    edge = 1e-3 * max(8, int(np.ceil((1.2 * n) ** (1 / 3))))
    h = sedi.Sedi(default_params(hi=(edge, edge, 2 * edge), ncell=(8, 8, 8), wall_hi=(0, 0, 0)))
    x = lattice_bed(n, edge, 0.5e-3, 3, jitter=2e-4, spacing=1.0)
    g = np.random.default_rng(n)
    h.set_particles(x, 0.01 * g.normal(size=(n, 3)), g.normal(size=(n, 3)), np.full(n, 0.5e-3), np.full(n, 2500.0))
    return h


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513])
def test_forces_on_host_equal_device_outputs(n):
    h = handle(n)
    names = ("contact", "lub", "fluid", "torque")
    f = h.compute_forces()
    dev = [torch.full((n, 3), 7.0, dtype=torch.float64, device="cuda") for _ in names]
    h._check(sedi.lib().sedi_compute_forces(h.h, 0, *(t.data_ptr() for t in dev), 1))
    for k, t in zip(names, dev):
        np.testing.assert_array_equal(f[k], t.cpu().numpy())
    one = np.full((n, 3), 7.0)  # one output alone
    h._check(sedi.lib().sedi_compute_forces(h.h, 0, None, None, one.ctypes.data, None, 0))
    np.testing.assert_array_equal(one, f["fluid"])


def test_large_outputs_into_untouched_pages():
    """Four 24 MB arrays that the allocator gives back to the system and takes again each time:
    mapping their pages on the host takes 2 ms, from the GPU's side 60.  The call may take
    ten times what it takes into arrays in place (a page fault costs what 64 KB of copy do)."""
    n = 1_000_000
    h = handle(n)
    for _ in range(3):  # the allocator's threshold for memory from the system rises to this size
        a = [np.ones((n, 3)) for _ in range(4)]
        del a

    def timed(f):
        t = []
        for _ in range(5):
            t0 = time.perf_counter()
            f()
            t.append(time.perf_counter() - t0)
        return float(np.median(t))

    fresh = timed(h.compute_forces)
    out = [np.ones((n, 3)) for _ in range(4)]
    kept = timed(lambda: h._check(sedi.lib().sedi_compute_forces(h.h, 0, *(a.ctypes.data for a in out), 0)))
    assert fresh <= 10.0 * kept, (fresh, kept)
    f = h.compute_forces()
    for k, a in zip(("contact", "lub", "fluid", "torque"), out):
        np.testing.assert_array_equal(f[k], a)


def test_device_output_that_is_too_small_is_refused():
    """A device buffer smaller than the output is refused by the copy to it, as a host check: no
    kernel writes past its end.  The bytes behind it, in the same 2 MB page, stay."""
    cudart = ctypes.CDLL(next(line.split()[-1] for line in open("/proc/self/maps") if "libcudart.so" in line))

    def malloc(size):
        p = ctypes.c_void_p()
        assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        return p.value

    n = 1000
    h = handle(n)
    C = h.C
    short = 24 * n - 8192
    page = 2 << 20
    p = malloc(short)
    if p % page + 24 * n + 24 * C > page:
        pytest.skip("the buffer ends its page")
    for call in (lambda: sedi.lib().sedi_get_particles(h.h, 0, p, None, None, None, 1),
                 lambda: sedi.lib().sedi_average(h.h, 0, None, p - p % 8 + short // 8 * 8 - 8, None, 1)):
        with pytest.raises(sedi.SediError) as e:
            h._check(call())
        assert e.value.code == -3
    h.step(2)  # the handle and the context are in order
    want = h.get_particles()[0]
    q = malloc(24 * n)
    h._check(sedi.lib().sedi_get_particles(h.h, 0, q, None, None, None, 1))
    got = np.zeros((n, 3))
    assert cudart.cudaMemcpy(ctypes.c_void_p(got.ctypes.data), ctypes.c_void_p(q), ctypes.c_size_t(24 * n), 2) == 0
    np.testing.assert_array_equal(got, want)
    for r in (p, q):
        cudart.cudaFree(ctypes.c_void_p(r))
