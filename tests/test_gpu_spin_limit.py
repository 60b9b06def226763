"""The limit of the smoother's waits can be lowered and never raised: a value beyond 32 bits
counts as the default (cut to 32 bits it would be 0, and the first wait would run out)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params, random_fields  # noqa: E402


@pytest.mark.parametrize("limit", ["4294967296", "8589934593", "9223372036854775807"])
@pytest.mark.parametrize("form", ["split", "fp64"])
def test_large_limit_is_the_default(monkeypatch, form, limit):
    prm = dict(default_params(hi=(96e-3, 96e-3, 24e-3), ncell=(96, 96, 24), wall_hi=(0, 0, 1),
                              bandwidth=(2e-3, 2e-3, 1.5e-3)), precision_form=form)
    phi = random_fields(prm["ncell"], 2, seed=61)
    want, _ = sedi.Sedi(prm).smooth(phi)
    monkeypatch.setenv("SEDI_BARRIER_SPIN_LIMIT", limit)
    out, _ = sedi.Sedi(prm).smooth(phi)
    np.testing.assert_array_equal(out, want)
