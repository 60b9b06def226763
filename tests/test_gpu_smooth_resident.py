"""The resident smoothing solver at the edges of its cuts: bricks of one cell, chunks that a
brick ends inside, one CTA, a cluster, whole-chip groups with and without a cut across z,
wrapped and closed axes, both pseudo-time schemes, guesses, a graded mesh; and many
fields of different meshes through one cluster."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as orc  # noqa: E402
from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params, ensemble_case, random_fields  # noqa: E402


def mesh(ncell, periodic, scheme=0, grading=1.0):
    return default_params(hi=tuple(1e-3 * n for n in ncell), ncell=ncell, periodic=periodic, wall_lo=(0, 0, 0),
                          wall_hi=(0, 0, 0), bandwidth=(2.5e-3, 2e-3, 1.5e-3), tau_scheme=scheme,
                          z_grading=grading)


# 1e-7 of the largest value: both sides stop at a residual of 1e-8 |b|, and |A^-1| = 1
@pytest.mark.parametrize("form", ["split", "fp64"])
@pytest.mark.parametrize("ncell,periodic,scheme,grading", [
    ((1, 1, 1), (1, 1, 0), 0, 1.0), ((5, 7, 9), (1, 0, 1), 1, 1.0), ((3, 1, 41), (0, 1, 0), 0, 1.0),
    ((70, 2, 3), (1, 1, 1), 0, 1.0), ((13, 17, 6), (0, 0, 0), 1, 3.0), ((33, 31, 19), (1, 1, 0), 1, 2.0),
    ((37, 41, 45), (1, 1, 1), 0, 1.0), ((64, 32, 61), (0, 1, 1), 1, 1.0)])
def test_cluster_cuts_match_oracle(ncell, periodic, scheme, grading, form):
    prm = mesh(ncell, periodic, scheme, grading)
    phi = random_fields(ncell, 3, seed=21)
    phi[1] = 0.0  # a field that needs no step among others
    out, it = sedi.Sedi(dict(prm, precision_form=form)).smooth(phi)
    ref, _ = orc.Oracle(prm).smooth(phi)
    assert np.abs(out - ref).max() <= 1e-7 * max(np.abs(phi).max(), 1e-300)
    assert not out[1].any() and it[1] == 0


@pytest.mark.parametrize("ncell,periodic,scheme,grading", [
    ((53, 51, 49), (1, 1, 1), 0, 1.0), ((200, 90, 11), (1, 0, 0), 1, 2.0), ((40, 36, 101), (0, 0, 1), 1, 1.0),
    ((150, 101, 93), (1, 1, 0), 0, 1.0)])
def test_grid_cuts_match_oracle(ncell, periodic, scheme, grading):
    prm = mesh(ncell, periodic, scheme, grading)
    phi = random_fields(ncell, 2, seed=22)
    guess = 0.5 * phi + 0.01
    g, o = sedi.Sedi(dict(prm, precision_form="split")), orc.Oracle(prm)
    for kw in ({}, {"guess": guess}):
        out, _ = g.smooth(phi, **kw)
        ref, _ = o.smooth(phi, **kw)
        assert np.abs(out - ref).max() <= 1e-7 * np.abs(phi).max()


def test_many_meshes_share_a_cluster():
    """48 beds on 16^3 .. 48^3 meshes: 336 fields, so every cluster takes several, each of
    another brick layout; every bed smooths to the bits it has alone."""
    prm, beds = ensemble_case(n_beds=48, seed=91, n_min=300, n_max=3000)
    rng = np.random.default_rng(7)
    e = sedi.Sedi(dict(prm, n_beds=len(beds), precision_form="split"))
    for b, bd in enumerate(beds):
        p = bd["parts"]
        p["v"] = rng.normal(0.0, 0.05, p["x"].shape)
        e.set_bed(b, bd["lo"], bd["hi"], bd["ncell"])
        e.set_particles(p["x"], p["v"], p["w"], p["d"], p["rho"], bed=b)
    e.average_inplace()
    for b, bd in enumerate(beds):
        p = bd["parts"]
        g = sedi.Sedi(dict(prm, lo=bd["lo"], hi=bd["hi"], ncell=bd["ncell"], precision_form="split"))
        g.set_particles(p["x"], p["v"], p["w"], p["d"], p["rho"])
        for one, many in zip(g.average(), e.average(bed=b)):
            assert np.array_equal(one, many), b
        g.close()
