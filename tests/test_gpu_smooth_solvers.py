"""The smoothing solvers against each other.  In FP32 words no bit of a result depends on which
of them takes a mesh: the on-chip solver against the cluster solver (meshes of one CTA) and
the streaming one (meshes beyond a cluster).  The streaming solver, which large and flat
meshes still take, against the oracle, and its grid barrier's wait running out."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as orc  # noqa: E402
from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import default_params, random_fields  # noqa: E402

ETIMEOUT = -8


def mesh(ncell, periodic, scheme=0, grading=1.0):
    return default_params(hi=tuple(1e-3 * n for n in ncell), ncell=ncell, periodic=periodic, wall_lo=(0, 0, 0),
                          wall_hi=(0, 0, 0), bandwidth=(2.5e-3, 2e-3, 1.5e-3), tau_scheme=scheme,
                          z_grading=grading)


def handles(monkeypatch, prm, form):
    on = sedi.Sedi(dict(prm, precision_form=form))
    monkeypatch.setenv("SEDI_SMOOTH_RESIDENT", "0")
    off = sedi.Sedi(dict(prm, precision_form=form))
    monkeypatch.delenv("SEDI_SMOOTH_RESIDENT")
    return on, off


# one CTA on chip against the cluster solver, then whole-chip groups against the streaming one
@pytest.mark.parametrize("form", ["split", "plain"])
@pytest.mark.parametrize("ncell,periodic,scheme,grading", [
    ((1, 1, 1), (1, 1, 0), 0, 1.0), ((5, 7, 9), (1, 0, 1), 1, 1.0), ((13, 17, 6), (0, 0, 0), 1, 3.0),
    ((16, 16, 32), (1, 1, 1), 0, 1.0), ((10, 10, 20), (1, 1, 0), 0, 2.0), ((31, 33, 8), (0, 1, 0), 1, 1.0),
    ((53, 51, 49), (1, 1, 1), 0, 1.0), ((200, 90, 11), (1, 0, 0), 1, 2.0), ((40, 36, 101), (0, 0, 1), 1, 1.0),
    ((96, 96, 24), (1, 1, 0), 0, 3.0), ((120, 120, 4), (0, 1, 1), 1, 1.0), ((150, 101, 93), (1, 1, 0), 0, 1.0)])
def test_same_bits_from_every_solver(monkeypatch, ncell, periodic, scheme, grading, form):
    on, off = handles(monkeypatch, mesh(ncell, periodic, scheme, grading), form)
    phi = random_fields(ncell, 4, seed=17)
    phi[2] = 0.0
    for kw in ({}, {"guess": 0.5 * phi + 0.01}):
        a, ia = on.smooth(phi, **kw)
        b, ib = off.smooth(phi, **kw)
        np.testing.assert_array_equal(a, b)
        np.testing.assert_array_equal(ia, ib)


# 1e-7 of the largest value: both sides stop at a residual of 1e-8 |b| (plain form: 2e-6, and
# FP32 words), and |A^-1| = 1
@pytest.mark.parametrize("form,tol", [("split", 1e-7), ("fp64", 1e-7), ("plain", 2e-5)])
@pytest.mark.parametrize("ncell,periodic,scheme,grading", [
    ((96, 96, 24), (1, 1, 0), 0, 3.0), ((96, 96, 24), (1, 1, 0), 1, 1.0), ((100, 100, 1), (1, 0, 0), 0, 1.0),
    ((53, 51, 49), (1, 1, 1), 1, 1.0)])
def test_streaming_solver_matches_oracle(monkeypatch, ncell, periodic, scheme, grading, form, tol):
    prm = mesh(ncell, periodic, scheme, grading)
    off = handles(monkeypatch, prm, form)[1]
    phi = random_fields(ncell, 2, seed=23)
    out, _ = off.smooth(phi)
    ref, _ = orc.Oracle(prm).smooth(phi)
    assert np.abs(out - ref).max() <= tol * np.abs(phi).max()


def test_streaming_barrier_timeout_is_reported_and_handle_recovers(monkeypatch):
    """A poll limit of 1 lets the first wait at the grid barrier run out; the call reports it, and
    the handle's state and a fresh handle are usable."""
    prm = mesh((96, 96, 24), (1, 1, 0))
    phi = random_fields(prm["ncell"], 2, seed=61)
    monkeypatch.setenv("SEDI_SMOOTH_RESIDENT", "0")
    want, _ = sedi.Sedi(dict(prm, precision_form="split")).smooth(phi)
    monkeypatch.setenv("SEDI_BARRIER_SPIN_LIMIT", "1")
    g = sedi.Sedi(dict(prm, precision_form="split"))
    monkeypatch.delenv("SEDI_BARRIER_SPIN_LIMIT")
    with pytest.raises(sedi.SediError) as e:
        g.smooth(phi)
    assert e.value.code == ETIMEOUT
    x = np.array([[0.02, 0.03, 0.01], [0.05, 0.06, 0.012]])
    g.set_particles(x, np.zeros((2, 3)), np.zeros((2, 3)), np.full(2, 1e-3), np.full(2, 2500.0))
    g.step(3)
    g.sync()
    out, _ = sedi.Sedi(dict(prm, precision_form="split")).smooth(phi)
    np.testing.assert_array_equal(out, want)


# whole-chip groups from one cell a brick up, cuts that change with the number of fields, and
# meshes of one cell across
@pytest.mark.parametrize("ncell,periodic,scheme,grading", [
    ((5, 7, 9), (1, 0, 1), 1, 1.0), ((8, 8, 8), (1, 1, 0), 0, 1.0), ((13, 17, 6), (0, 0, 0), 1, 3.0),
    ((19, 15, 31), (1, 1, 0), 0, 1.0), ((70, 2, 3), (1, 1, 1), 0, 1.0), ((3, 1, 41), (0, 1, 0), 0, 1.0),
    ((37, 41, 45), (1, 1, 0), 1, 2.0), ((53, 51, 49), (1, 1, 1), 0, 1.0), ((100, 100, 1), (0, 1, 0), 1, 1.0)])
def test_same_fp64_bits_from_every_solver_and_cut(monkeypatch, ncell, periodic, scheme, grading):
    on, off = handles(monkeypatch, mesh(ncell, periodic, scheme, grading), "fp64")
    phi = random_fields(ncell, 8, seed=19)
    phi[2] = 0.0
    want, steps = off.smooth(phi)
    for nf in (8, 7, 2, 1):
        out, it = on.smooth(phi[:nf])
        np.testing.assert_array_equal(out, want[:nf])
        np.testing.assert_array_equal(it, steps[:nf])


def test_chip_is_cut_for_the_fields_asked_for():
    """FP64 on 64 x 32 x 64: seven fields side by side take a seventh of the chip each, so one
    field alone on such a seventh would take as long as seven, and eight twice as long.
    Cut for its own number a call measured 0.23 and 1.23 times the time of seven."""
    h = sedi.Sedi(dict(mesh((64, 32, 64), (1, 1, 0)), precision_form="fp64"))
    x = torch.rand((8, h.C), dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    it = np.zeros(8, np.int32)

    def timed(nf):
        t = []
        for _ in range(6):
            t0 = time.perf_counter()
            h._check(sedi.lib().sedi_smooth(h.h, 0, nf, x.data_ptr(), y.data_ptr(), None, it.ctypes.data, 1))
            t.append(time.perf_counter() - t0)
        return float(np.median(t))

    t1, t7, t8 = timed(1), timed(7), timed(8)
    assert t1 <= 0.5 * t7 and t8 <= 1.6 * t7, (t1, t7, t8)
