"""What a small handle costs beside its work: no memory is pinned for a handle that is created,
loaded and released, since that takes a fifth of the whole."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import small_case  # noqa: E402


def median_time(f, reps=15):
    t = []
    for _ in range(reps):
        t0 = time.perf_counter()
        f()
        t.append(time.perf_counter() - t0)
    return float(np.median(t))


def test_first_load_costs_little_more_than_a_reload():
    """A first load differs from a reload of the same particles by its allocations, a tenth of
    what creating and releasing the handle takes; pinning memory made it more than
    that whole.  Both times include the same copies and list build; medians, with room for a busy host."""
    prm, parts = small_case()
    args = [parts[k][:100] for k in ("x", "v", "w", "d", "rho")]
    bare = median_time(lambda: sedi.Sedi(prm).close())

    def whole():
        h = sedi.Sedi(prm)
        h.set_particles(*args)
        h.close()

    whole()
    first = median_time(whole) - bare
    h = sedi.Sedi(prm)
    h.set_particles(*args)
    again = median_time(lambda: h.set_particles(*args))
    assert first - again <= 0.75 * bare, (bare, first, again)
