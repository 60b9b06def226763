"""The work that a user of this framework has it do, as a list of timed cases.

Every case goes through the public entry points: the binding `sedi` (and, where a
result is wanted on the device, the C ABI behind it with its device-memory flag).
A case is a dict of plain values; `kind` says which call it stands for:

* step      one fluid step of a coupled run: DEM substeps, the averaged fields back, and
            the particle state (what a coupling code takes over)
* ensemble  the same for many independent beds of uneven size in one handle
* average   the averaging of a bed that was just loaded (a restart, a diagnostic)
* smooth    diffusion smoothing of a caller's own fields, without a handle
* filter    the same through a handle (large meshes, BDF2, graded meshes)
* load      new particles into a handle and its neighbour lists back (each substep of a
            decomposed run, a restart)
* forces    the forces of a state, kind by kind (diagnostics, validation)
* train     training of the warm-start network on pairs of fields
* infer     that network applied to a field

Beds are made as the framework's own workloads make them (a settled periodic block
tiled over the floor, workloads.settled_bed), from smaller blocks so that another seed
is another bed in under a second.
"""
import math

import numpy as np
import torch

from paper_1601_03801_gb300 import sedi
from paper_1601_03801_gb300.workloads import (default_params, ensemble_case, lattice_bed, lognormal_d,
                                              settled_bed, small_case, uniform_d)

DEV = "cuda"
BLOCK = 2e-3  # edge of a settled block's footprint (m)


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest configuration: 1,000 spheres in quiescent water, 20 substeps a
        # fluid step; launches and latency
        dict(name="step_small", kind="step", bed="small", n=1000, form="split", substeps=20),
        # the sheared sediment bed: 200,000 lognormal spheres, 64 x 32 x 64 mesh
        dict(name="step_bed", kind="step", bed="lognormal", n=200_000, tx=32, ty=16, height=64e-3,
             nx=64, ny=32, nz=64, form="split", substeps=20),
        # the headline: 10,000,000 spheres, 256 x 128 x 64 mesh
        dict(name="step_large", kind="step", bed="uniform", n=10_000_000, tx=200, ty=100,
             height=100e-3, nx=256, ny=128, nz=64, form="split", substeps=20),
        # the FP64 parity form, as it is used to check a run: a small bed, odd count and mesh
        dict(name="step_fp64", kind="step", bed="uniform", n=20_011, tx=9, ty=7, height=30e-3,
             nx=19, ny=15, nz=31, form="fp64", substeps=10),
        # the plain FP32 form (the comparison baseline) on a middle-sized bed
        dict(name="step_plain", kind="step", bed="uniform", n=500_003, tx=40, ty=26, height=50e-3,
             nx=81, ny=51, nz=48, form="plain", substeps=20),
        # parameter studies: many beds of 2,000 to 50,000 spheres, 16^3 to 48^3 meshes
        dict(name="ensemble", kind="ensemble", beds=48, mix=1601038014, n_min=2000, n_max=50_000,
             substeps=20),
        # averaging on the fine 128 x 64 x 128 mesh of the warm-start runs
        dict(name="average_fine", kind="average", bed="lognormal", n=200_000, tx=32, ty=16,
             height=64e-3, nx=128, ny=64, nz=128, form="split"),
        # a field on a small mesh of an odd size, smoothed without a handle
        dict(name="smooth_odd", kind="smooth", fields=4, nx=37, ny=41, nz=45, scheme=0, form="split"),
        # all seven fields of the large bed's mesh, second-order pseudo-time, graded mesh
        dict(name="filter_large", kind="filter", fields=7, nx=256, ny=128, nz=64, scheme=1,
             grading=2.0, form="split"),
        # new particles into a handle and the lists back
        dict(name="load_bed", kind="load", bed="lognormal", n=200_000, tx=32, ty=16, height=64e-3,
             form="split"),
        # the forces of a state
        dict(name="forces_bed", kind="forces", bed="lognormal", n=100_003, tx=17, ty=16,
             height=64e-3, nx=34, ny=32, nz=64, form="split"),
        # training of the warm-start network on the sheared bed's mesh
        dict(name="train", kind="train", nx=64, ny=32, nz=64, pairs=4, steps=8),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "ensemble", "average", "smooth", "filter", "load",
                       "forces", "train", "infer"])
    if kind == "ensemble":
        return dict(kind=kind, beds=rng.randint(2, 48), mix=rng.randint(1, 1 << 30), n_min=rng.randint(500, 3000),
                    n_max=rng.randint(6000, 50_000), substeps=rng.randint(1, 20))
    if kind in ("smooth", "filter"):
        c = dict(kind=kind, fields=rng.randint(1, 7), scheme=rng.randint(0, 1),
                 form=rng.choice(["split", "split", "split", "plain", "fp64"]))
        if kind == "smooth":
            cells = _logint(rng, 2000, 120_000)
        else:
            cells = _logint(rng, 20_000, 2_000_000 if c["form"] != "fp64" else 300_000)
            c["grading"] = rng.choice([1.0, 1.0, rng.uniform(1.5, 4.0)])
        e = cells ** (1.0 / 3.0)
        c["nx"] = max(5, int(e * rng.uniform(0.6, 1.6)))
        c["ny"] = max(5, int(e * rng.uniform(0.6, 1.6)))
        c["nz"] = max(5, cells // (c["nx"] * c["ny"]))
        return c
    if kind in ("train", "infer"):
        return dict(kind=kind, nx=rng.randint(12, 72), ny=rng.randint(12, 48), nz=rng.randint(12, 64),
                    pairs=rng.randint(1, 4), steps=rng.randint(1, 8))
    form = "split"
    if kind == "step":
        form = rng.choice(["split", "split", "split", "plain", "fp64"])
    top = {"step": {"split": 4_000_000, "plain": 2_000_000, "fp64": 30_000}[form], "average": 1_000_000,
           "load": 400_000, "forces": 150_000}[kind]
    n = _logint(rng, 1000, top)
    per = rng.randint(120, 500)
    tiles = max(4, -(-n // per))
    tx = max(2, int(round(math.sqrt(tiles) * rng.uniform(0.7, 1.5))))
    ty = max(2, -(-tiles // tx))
    c = dict(kind=kind, bed=rng.choice(["uniform", "lognormal"]), n=n, tx=tx, ty=ty,
             height=rng.uniform(20e-3, 60e-3), form=form)
    if kind == "step":
        c["substeps"] = rng.randint(1, 20)
    if kind != "load":
        c.update(nx=max(4, int(tx * rng.uniform(1.0, 2.5))), ny=max(4, int(ty * rng.uniform(1.0, 2.5))),
                 nz=rng.randint(12, 64))
    return c


# ---------------------------------------------------------------- inputs
def _bed(case, seed):
    """Particles of a settled bed (host arrays, as a program reads them from a file)."""
    n, tiles = case["n"], case["tx"] * case["ty"]
    nb = -(-n // tiles)
    uniform = case["bed"] == "uniform"
    dsample = uniform_d(0.4e-3, 0.6e-3) if uniform else lognormal_d(0.5e-3, 0.1)
    x, d = settled_bed(nb, (1, 1), (BLOCK, BLOCK), dsample, 4 * seed + (1 if uniform else 2), iters=1500)
    off = np.stack(np.meshgrid(np.arange(case["tx"]) * BLOCK, np.arange(case["ty"]) * BLOCK, [0.0],
                               indexing="ij"), -1).reshape(-1, 1, 3)
    X = (off + x[None]).reshape(-1, 3)
    D = np.tile(d, tiles)
    L = (case["tx"] * BLOCK, case["ty"] * BLOCK, max(case["height"], 1.05 * float(x[:, 2].max() + d.max())))
    for a in range(2):
        X[:, a] = np.minimum(X[:, a], np.nextafter(L[a], 0.0))
    if len(X) > n:  # the bed's surface is where spheres are missing
        keep = np.ones(len(X), bool)
        keep[np.argpartition(X[:, 2], n)[n:]] = False
        X, D = X[keep], D[keep]
    g = torch.Generator(device=DEV).manual_seed(seed)
    v = (3e-3 * torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)).cpu().numpy()
    w = (2.0 * torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)).cpu().numpy()
    return L, dict(x=X, v=v, w=w, d=D, rho=np.full(n, 2500.0))


def _flow(nc, L, seed):
    """Mean flow of 0.3 m/s plus filtered noise of rms 0.03 m/s, and U . grad U."""
    g = torch.Generator(device=DEV).manual_seed(seed + 7)
    nx, ny, nz = nc
    f = torch.fft.fftn(torch.randn(3, nz, ny, nx, generator=g, device=DEV, dtype=torch.float64), dim=(1, 2, 3))
    for ax, m in ((1, nz), (2, ny), (3, nx)):
        k = torch.fft.fftfreq(m, device=DEV, dtype=torch.float64)
        shape = [1, 1, 1, 1]
        shape[ax] = m
        f = f * torch.exp(-2.0 * (math.pi * k * 2.0) ** 2).view(shape)
    U = torch.fft.ifftn(f, dim=(1, 2, 3)).real
    U = 0.03 * U / U.std(dim=(1, 2, 3), keepdim=True)
    U[0] += 0.3
    DU = torch.zeros_like(U)
    for a, ax in ((0, 3), (1, 2), (2, 1)):
        DU += U[a] * (torch.roll(U, -1, ax) - torch.roll(U, 1, ax)) * (0.5 * nc[a] / L[a])
    flat = lambda t: t.permute(1, 2, 3, 0).reshape(-1, 3).contiguous()  # noqa: E731
    return flat(U), flat(DU)


def _params(case, L):
    return default_params(hi=tuple(L), wall_hi=(0, 0, 0), bandwidth=(1.5e-3,) * 3,
                          ncell=(case.get("nx", 8), case.get("ny", 8), case.get("nz", 8)))


def _mesh_params(case):
    """Parameters of a smoothing alone: 1 mm cells, anisotropic bandwidths of 2 to 3 mm."""
    nc = (case["nx"], case["ny"], case["nz"])
    return default_params(hi=tuple(1e-3 * n for n in nc), ncell=nc, wall_hi=(0, 0, 0),
                          bandwidth=(3e-3, 3e-3, 2e-3), tau_scheme=case["scheme"],
                          z_grading=case.get("grading", 1.0))


def _fields(nf, cells, seed):
    """Non-negative fields with empty cells, as a deposition leaves them."""
    g = torch.Generator(device=DEV).manual_seed(seed + 3)
    f = torch.rand(nf, cells, generator=g, device=DEV, dtype=torch.float64)
    return torch.where(torch.rand(nf, cells, generator=g, device=DEV) < 0.5, torch.zeros_like(f), f)


def _net(case, seed):
    """Network weights and training pairs: smooth fields of order one."""
    rng = np.random.default_rng(seed)
    nc = (case["nx"], case["ny"], case["nz"])
    C = nc[0] * nc[1] * nc[2]
    w = np.concatenate([rng.normal(0, (2.0 / (27 * 4)) ** 0.5, 32 * 4 * 27), rng.normal(0, 0.05, 32),
                        rng.normal(0, (2.0 / (27 * 32)) ** 0.5, 32 * 32 * 27), rng.normal(0, 0.05, 32),
                        rng.normal(0, (1.0 / (27 * 32)) ** 0.5, 4 * 32 * 27), rng.normal(0, 0.05, 4)])
    x = torch.cat([_flow(nc, (1.0, 1.0, 1.0), seed + 11 * k)[0].T for k in range(2 * case["pairs"])])
    x = ((x - x.mean(1, keepdim=True)) / x.std(1, keepdim=True))
    x = torch.cat([x, x[:2 * case["pairs"]] * x[2 * case["pairs"]:4 * case["pairs"]]])[:8 * case["pairs"]]
    x = x.reshape(2, case["pairs"], 4, C).cpu().numpy().copy()
    return w, x[0], 0.3 * x[1]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "smooth":
        p = dict(_mesh_params(case), precision_form=case["form"])
        phi = _fields(case["fields"], case["nx"] * case["ny"] * case["nz"], seed)
        return dict(kind=kind, p=p, phi=phi, out=torch.empty_like(phi))
    if kind == "filter":
        h = sedi.Sedi(dict(_mesh_params(case), precision_form=case["form"]))
        phi = _fields(case["fields"], h.C, seed)
        torch.cuda.synchronize()
        return dict(kind=kind, h=h, phi=phi, out=torch.empty_like(phi), nf=case["fields"])
    if kind in ("train", "infer"):
        w, x, t = _net(case, seed)
        h = sedi.Sedi(default_params(ncell=(case["nx"], case["ny"], case["nz"])))
        h.cnn_set_params(w)
        return dict(kind=kind, h=h, w=w, x=x, t=t, steps=case["steps"])
    if kind == "ensemble":
        # the beds' sizes belong to the case (`mix`), their spheres to the seed
        prm, beds = ensemble_case(case["beds"], seed=case["mix"], n_min=case["n_min"], n_max=case["n_max"])
        h = sedi.Sedi(dict(prm, n_beds=len(beds)))
        g = np.random.default_rng(seed)
        for b, bd in enumerate(beds):
            h.set_bed(b, bd["lo"], bd["hi"], bd["ncell"])
            p = bd["parts"]
            p["x"] = lattice_bed(len(p["d"]), bd["hi"][0], 0.5e-3, seed + 1 + b, jitter=2e-4, spacing=1.0)
            h.set_particles(p["x"], 1e-3 * g.normal(size=p["x"].shape), g.normal(size=p["x"].shape),
                            p["d"], p["rho"], bed=b)
            h.set_fluid(U=bd["U"], bed=b)
        n = [len(bd["parts"]["x"]) for bd in beds]
        c = [int(np.prod(bd["ncell"])) for bd in beds]
        x = torch.empty(sum(n), 3, dtype=torch.float64, device=DEV)
        eps = torch.empty(sum(c), dtype=torch.float64, device=DEV)
        us = torch.empty(sum(c), 3, dtype=torch.float64, device=DEV)
        s = dict(kind=kind, h=h, x=x, xs=x.split(n), eps=eps, es=eps.split(c), us=us, uss=us.split(c),
                 k=case["substeps"])
        h.step(200)  # a run under way: springs formed, launch shapes tuned
        h.step(case["substeps"])
        h.average_inplace()
        return s
    if case["bed"] == "small":
        prm, parts = small_case(seed, parity_addon=True)
    else:
        L, parts = _bed(case, seed)
        prm = _params(case, L)
    if kind == "load":
        h = sedi.Sedi(dict(prm, precision_form=case["form"]))
        return dict(kind=kind, h=h, parts=parts, off=np.zeros(case["n"] + 1, dtype=np.int64),
                    ids=np.zeros(16 * case["n"], dtype=np.int64))
    h = sedi.Sedi(dict(prm, precision_form=case["form"]))
    h.set_particles(parts["x"], parts["v"], parts["w"], parts["d"], parts["rho"])
    if case["bed"] != "small":
        U, DU = _flow(prm["ncell"], prm["hi"], seed)
        torch.cuda.synchronize()
        h.set_fluid(U=U, DUDt=DU)
    out = lambda rows, *w: torch.zeros(rows, *w, dtype=torch.float64, device=DEV)  # noqa: E731
    s = dict(kind=kind, h=h, k=case.get("substeps", 0))
    if kind != "forces":
        s.update(eps=out(h.C), us=out(h.C, 3), f=out(h.C, 3))
    if kind == "step":
        s.update(x=out(h.n, 3), v=out(h.n, 3), w=out(h.n, 3))
        torch.cuda.synchronize()
        if case["form"] != "fp64":  # a run under way: springs formed, launch shapes tuned
            h.step(200)
        h.step(case["substeps"])
        h.average(s["eps"], s["us"], s["f"])
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _averaged(s):
    """The averaged fields, the velocity as momentum per volume (a cell without spheres
    has no velocity: there it is a quotient of rounding errors)."""
    return {"eps": s["eps"], "mom": s["us"] * s["eps"][:, None]}


def run(s):
    kind, h = s["kind"], s.get("h")
    if kind == "step":
        h.step(s["k"])
        h.average(s["eps"], s["us"], s["f"])
        h._check(sedi.lib().sedi_get_particles(h.h, 0, s["x"].data_ptr(), s["v"].data_ptr(),
                                               s["w"].data_ptr(), None, sedi.MEM_DEVICE))
        return dict(_averaged(s), **{q: s[q] for q in ("f", "x", "v", "w")})
    if kind == "ensemble":
        h.step(s["k"])
        h.average_inplace()
        for b in range(h.n_beds):
            h.average(s["es"][b], s["uss"][b], bed=b)
            h.get_positions(s["xs"][b], bed=b)
        return dict(_averaged(s), x=s["x"])
    if kind == "average":
        h.average(s["eps"], s["us"], s["f"])
        return dict(_averaged(s), f=s["f"])
    if kind == "smooth":
        sedi.smooth_static(s["p"], s["phi"], s["out"])
        return s["out"]
    if kind == "filter":
        h._check(sedi.lib().sedi_smooth(h.h, 0, s["nf"], s["phi"].data_ptr(), s["out"].data_ptr(), None,
                                        None, sedi.MEM_DEVICE))
        return s["out"]
    if kind == "load":
        p = s["parts"]
        h.set_particles(p["x"], p["v"], p["w"], p["d"], p["rho"])
        h._check(sedi.lib().sedi_get_neighbors(h.h, 0, s["off"].ctypes.data, s["ids"].ctypes.data,
                                               len(s["ids"])))
        return {"offsets": s["off"], "ids": s["ids"]}
    if kind == "forces":
        return h.compute_forces()
    # the network computes in FP32 words: the binding's float64 arrays only carry them
    if kind == "train":
        h.cnn_set_params(s["w"])
        losses = h.cnn_train(s["x"], s["t"], s["steps"], lr=1e-3)
        return {"losses": losses.astype(np.float32), "weights": h.cnn_get_params().astype(np.float32)}
    return h.cnn_forward(s["x"][0]).astype(np.float32)


# ---------------------------------------------------------------- least work
def work(case):
    kind = case["kind"]
    if kind in ("train", "infer"):
        C = case["nx"] * case["ny"] * case["nz"]
        macs = 27 * (4 * 32 + 32 * 32 + 32 * 4) * C
        if kind == "infer":
            return {"bytes": 64 * C, "flops": 2 * macs}
        # forward, weight gradients, and the data gradients of layers 2 and 3
        steps = 3 * macs - 27 * 4 * 32 * C
        return {"bytes": 64 * C * case["pairs"], "flops": 2 * steps * case["steps"]}
    if kind in ("smooth", "filter"):
        return {"bytes": 16 * case["fields"] * case["nx"] * case["ny"] * case["nz"], "flops": 0}
    if kind == "ensemble":
        n = case["beds"] * (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        return {"bytes": n * ((172 + 4 * 6 + 36 * 3) * case["substeps"] + 96 + 24), "flops": 0}
    n = case["n"]
    C = case["nx"] * case["ny"] * case["nz"] if "nx" in case else 2000
    if kind == "load":  # 11 words in, offsets and about 10 partners a sphere out
        return {"bytes": n * (88 + 8 + 80), "flops": 0}
    if kind == "forces":  # state, lists and mesh in, four vectors out
        return {"bytes": n * (72 + 16 + 40 + 96) + 32 * C, "flops": 0}
    if kind == "average":  # position, velocity, acceleration, radius in; seven fields out
        return {"bytes": n * 72 + 56 * C, "flops": 0}
    # a substep: state read and written, radius, acceleration, about 10 listed partners
    # and 5 springs a sphere, the mesh fields; then the averaging
    w = {"split": 172 + 40 + 180, "plain": 100 + 40 + 90, "fp64": 184 + 40 + 240}[case["form"]]
    return {"bytes": (n * w + 40 * C) * case["substeps"] + n * 72 + 56 * C + n * 72, "flops": 0}


# ---------------------------------------------------------------- in 64 bits
def _modes(n, coef, periodic, edges=None):
    """Eigenvectors and values of -coef L on one axis (the finite-volume Laplacian,
    periodic or with zero-flux ends, on cells between `edges` if given), and the cell
    weights that make it symmetric."""
    h = torch.ones(n, dtype=torch.float64) if edges is None else edges[1:] - edges[:-1]
    dist = torch.ones(n, dtype=torch.float64)
    if edges is not None:
        zc = 0.5 * (edges[1:] + edges[:-1])
        dist[:-1] = zc[1:] - zc[:-1]
    A = torch.zeros(n, n, dtype=torch.float64)
    for k in range(n if periodic and n > 1 else n - 1):
        j = (k + 1) % n
        A[k, k] += coef / (h[k] * dist[k])
        A[j, j] += coef / (h[j] * dist[k])
        A[k, j] -= coef / (h[k] * dist[k])
        A[j, k] -= coef / (h[j] * dist[k])
    r = h.sqrt()
    S = r[:, None] * A / r[None, :]
    lam, V = torch.linalg.eigh(0.5 * (S + S.T))
    return lam.to(DEV), V.to(DEV), r.to(DEV)


def _smoothed(p, phi):
    """n_tau implicit diffusion steps of phi [nf, C], solved in the operator's modes."""
    nx, ny, nz = p["ncell"]
    L = [p["hi"][a] - p["lo"][a] for a in range(3)]
    n_tau, rtol_free = p["n_tau"], phi.reshape(-1, nz, ny, nx)
    ops = []
    for a, n in enumerate((nx, ny, nz)):
        D = 0.25 * p["bandwidth"][a] ** 2 / n_tau
        if a == 2 and p["z_grading"] != 1.0:
            lr = math.log(p["z_grading"]) / (n - 1)
            k = torch.arange(n + 1, dtype=torch.float64)
            ops.append(_modes(n, D, False, L[2] * torch.expm1(k * lr) / math.expm1(n * lr)))
        else:
            ops.append(_modes(n, D / (L[a] / n) ** 2, bool(p["periodic"][a])))
    (lx, Vx, _), (ly, Vy, _), (lz, Vz, r) = ops
    f = rtol_free * r.view(-1, 1, 1)
    f = torch.einsum("fzyx,xi->fzyi", f, Vx)
    f = torch.einsum("fzyi,yj->fzji", f, Vy)
    f = torch.einsum("fzji,zk->fkji", f, Vz)
    lam = lz.view(-1, 1, 1) + ly.view(1, -1, 1) + lx.view(1, 1, -1)
    prev, cur = None, f
    for m in range(n_tau):
        if p["tau_scheme"] == 0 or m == 0:
            prev, cur = cur, cur / (1.0 + lam)
        else:
            prev, cur = cur, (4.0 / 3.0 * cur - prev / 3.0) / (1.0 + 2.0 / 3.0 * lam)
    f = torch.einsum("fkji,zk->fzji", cur, Vz)
    f = torch.einsum("fzji,yj->fzyi", f, Vy)
    f = torch.einsum("fzyi,xi->fzyx", f, Vx) / r.view(-1, 1, 1)
    return f.reshape(phi.shape)


def _fluid_force(p, x, r, v, U, DU):
    """Drag, pressure gradient and added mass on spheres at rest in time (no lagged
    acceleration, no solid fraction yet)."""
    nx, ny, nz = p["ncell"]
    idx, fr = [], []
    for a, n in enumerate((nx, ny, nz)):
        s = (x[:, a] - p["lo"][a]) * (n / (p["hi"][a] - p["lo"][a])) - 0.5
        if p["periodic"][a]:
            k = s.floor()
            i0 = k.long() % n
            idx.append((i0, (i0 + 1) % n))
        else:
            s = s.clamp(0, n - 1)
            k = s.floor().clamp(max=n - 2)
            idx.append((k.long(), k.long() + 1))
        fr.append((1.0 - (s - k), s - k))
    uf, g = torch.zeros_like(x), torch.zeros_like(x)
    G = p["c_add"] * p["rho_f"] * DU - p["rho_f"] * torch.tensor(p["g"], dtype=torch.float64, device=DEV)
    for c in range(8):
        kx, ky, kz = c & 1, (c >> 1) & 1, c >> 2
        cell = (idx[2][kz] * ny + idx[1][ky]) * nx + idx[0][kx]
        wt = (fr[0][kx] * fr[1][ky] * fr[2][kz])[:, None]
        uf += wt * U[cell]
        g += wt * G[cell]
    d = 2.0 * r
    Vp = math.pi / 6 * d ** 3
    w = uf - v
    wm = w.norm(dim=1)
    Re = d * wm / p["nu_f"]
    vr = 0.5 * (1.0 - 0.06 * Re + ((0.06 * Re) ** 2 + 0.12 * Re + 1.0).sqrt())  # no solid fraction: A = B = 1
    cd = 0.63 * wm.sqrt() + 4.8 * (vr * p["nu_f"] / d).sqrt()
    return Vp[:, None] * g + (0.75 * Vp * p["rho_f"] * cd ** 2 / (vr ** 2 * d))[:, None] * w


def _pairs(p, x, cut):
    """Pairs within `cut`, each once: bins of that edge, sorted, every bin against half of
    its neighbours."""
    L = torch.tensor([p["hi"][a] - p["lo"][a] for a in range(3)], dtype=torch.float64, device=DEV)
    nb = [max(1, int(math.floor(float(L[a]) / cut))) for a in range(3)]
    nbt = torch.tensor(nb, device=DEV)
    c = torch.minimum((x / (L / nbt)).floor().long().clamp(min=0), nbt - 1)
    key = (c[:, 2] * nb[1] + c[:, 1]) * nb[0] + c[:, 0]
    order = key.argsort(stable=True)
    count = torch.bincount(key, minlength=nb[0] * nb[1] * nb[2])
    start = count.cumsum(0) - count
    out, per = [], torch.tensor(p["periodic"], device=DEV)
    for o in range(27):
        off = torch.tensor([o % 3 - 1, (o // 3) % 3 - 1, o // 9 - 1], device=DEV)
        t = c + off
        ok = (((t >= 0) & (t < nbt)) | (per > 0)).all(1)
        t = t % nbt
        tk = (t[:, 2] * nb[1] + t[:, 1]) * nb[0] + t[:, 0]
        for k in range(int(count.max())):
            i = (ok & (count[tk] > k)).nonzero()[:, 0]
            j = order[start[tk[i]] + k]
            i, j = i[i < j], j[i < j]
            dx = x[j] - x[i]
            dx = dx - per * L * (dx / L).round()
            near = (dx * dx).sum(1) < cut * cut
            out.append((i[near], j[near], dx[near]))
    return [torch.cat(q) for q in zip(*out)]


def _forces(p, parts, U, DU):
    """Contact (no contact history), lubrication and fluid force and contact torque."""
    t = lambda q: torch.from_numpy(np.ascontiguousarray(q)).to(DEV)  # noqa: E731
    x, v, w, r = t(parts["x"]), t(parts["v"]), t(parts["w"]), 0.5 * t(parts["d"])
    m = t(parts["rho"]) * math.pi / 6 * (2 * r) ** 3
    Es = p["E"] / (2 * (1 - p["poisson"] ** 2))
    Gs = p["E"] / (2 * (1 + p["poisson"])) / (2 * (2 - p["poisson"]))
    lne = math.log(p["restitution"])
    beta = lne / math.sqrt(lne ** 2 + math.pi ** 2)
    damp, mu6 = -2 * math.sqrt(5.0 / 6.0) * beta, 6 * math.pi * p["rho_f"] * p["nu_f"]
    fc, fl, tq = (torch.zeros_like(x) for _ in range(3))

    def touching(n, delta, Rs, ms, vrel):
        sq = (Rs * delta).sqrt()
        Sn, St = 2 * Es * sq, 8 * Gs * sq
        vn = (vrel * n).sum(1)
        vt = vrel - vn[:, None] * n
        fn = -(4.0 / 3.0) * Es * sq * delta - damp * (Sn * ms).sqrt() * vn
        ft = -(St * p["dt"] + damp * (St * ms).sqrt())[:, None] * vt
        cap = p["friction"] * fn.abs() / ft.norm(dim=1).clamp(min=1e-300)
        ft = ft * cap.clamp(max=1.0)[:, None]
        return fn[:, None] * n + ft, ft

    i, j, dx = _pairs(p, x, 1.1 * 2 * float(r.max()) * 1.0001)
    dist = dx.norm(dim=1)
    n, s = dx / dist[:, None], r[i] + r[j]
    delta = s - dist
    q = delta > 0
    a, b, nq, dq = i[q], j[q], n[q], delta[q]
    la, lb = (r[a] - 0.5 * dq)[:, None], (r[b] - 0.5 * dq)[:, None]
    vrel = v[a] - v[b] + torch.linalg.cross(la * w[a] + lb * w[b], nq)
    F, ft = touching(nq, dq, r[a] * r[b] / (r[a] + r[b]), m[a] * m[b] / (m[a] + m[b]), vrel)
    T = torch.linalg.cross(nq, ft)
    fc.index_add_(0, a, F).index_add_(0, b, -F)
    tq.index_add_(0, a, la * T).index_add_(0, b, lb * T)
    q = -delta < p["lub_h_out_frac"] * s
    a, b, nq = i[q], j[q], n[q]
    gap = torch.maximum(-delta[q], p["lub_h_in_frac"] * s[q])
    vn = ((v[a] - v[b]) * nq).sum(1)
    F = (-mu6 * (r[a] * r[b] / s[q]) ** 2 * vn / gap)[:, None] * nq
    fl.index_add_(0, a, F).index_add_(0, b, -F)
    # the floor
    n = torch.tensor([[0.0, 0.0, -1.0]], dtype=torch.float64, device=DEV)
    delta = r - (x[:, 2] - p["lo"][2])
    a = (delta > 0).nonzero()[:, 0]
    lev = (r[a] - 0.5 * delta[a])[:, None]
    nq = n.expand(len(a), 3)
    F, ft = touching(nq, delta[a], r[a], m[a], v[a] + torch.linalg.cross(lev * w[a], nq))
    fc[a] += F
    tq[a] += lev * torch.linalg.cross(nq, ft)
    a = (-delta < p["lub_h_out_frac"] * 2 * r).nonzero()[:, 0]
    gap = torch.maximum(-delta[a], p["lub_h_in_frac"] * 2 * r[a])
    fl[a] += (-mu6 * r[a] ** 2 * -v[a, 2] / gap)[:, None] * n
    return {"contact": fc, "lub": fl, "fluid": _fluid_force(p, x, r, v, U, DU), "torque": tq}


def _network(case, w, x, t, steps):
    """The network with its bfloat16 weights and activations, every sum in 64 bits; then
    `steps` Adam steps, and the losses."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    bf = lambda q: q.to(torch.float32).to(torch.bfloat16).to(torch.float64)  # noqa: E731
    shapes = [(32, 4, 3, 3, 3), (32,), (32, 32, 3, 3, 3), (32,), (4, 32, 3, 3, 3), (4,)]
    P, at = [], 0
    for s in shapes:
        k = int(np.prod(s))
        P.append(torch.tensor(w[at:at + k], device=DEV).float().double().reshape(s))
        at += k

    def pad(q, grads=False):  # periodic in x and y, zero outside in z
        q = torch.nn.functional.pad(q, (1, 1, 1, 1, 0, 0), mode="circular")
        return torch.nn.functional.pad(q, (0, 0, 0, 0, 1, 1))

    def unfold(q):  # [c, z, y, x] -> [c * 27, cells]
        q = pad(q[None])[0]
        u = q.unfold(1, nz, 1).unfold(2, ny, 1).unfold(3, nx, 1)
        return u.reshape(q.shape[0] * 27, -1)

    def conv(W, b, q):
        return (W.reshape(W.shape[0], -1) @ unfold(q) + b[:, None]).reshape(-1, nz, ny, nx)

    def back(W, g):  # data gradient: mirrored taps, weights transposed
        return conv(W.flip(2, 3, 4).transpose(0, 1), torch.zeros(W.shape[1], device=DEV, dtype=torch.float64), g)

    def forward(q):
        R = [bf(k) for k in P]
        a0 = bf(torch.tensor(q, device=DEV).reshape(4, nz, ny, nx))
        a1 = bf(conv(R[0], R[1], a0).clamp(min=0))
        a2 = bf(conv(R[2], R[3], a1).clamp(min=0))
        return R, a0, a1, a2, conv(R[4], R[5], a2)

    if not steps:
        return forward(x[0])[-1].reshape(4, -1)
    M, V, losses = [torch.zeros_like(q) for q in P], [torch.zeros_like(q) for q in P], []
    for k in range(steps):
        R, a0, a1, a2, y = forward(x[k % len(x)])
        e = y - torch.tensor(t[k % len(t)], device=DEV).reshape(y.shape)
        losses.append(float((e * e).mean()))
        g3 = 2 * e / e.numel()
        g2 = back(R[4], g3) * (a2 > 0)
        g1 = back(R[2], g2) * (a1 > 0)
        G = []
        for q, g, s in ((a0, g1, shapes[0]), (a1, g2, shapes[2]), (a2, g3, shapes[4])):
            g = g.reshape(g.shape[0], -1)
            G += [(g @ unfold(q).T).reshape(s), g.sum(1)]
        for q, g, m, v in zip(P, G, M, V):
            m.mul_(0.9).add_(g, alpha=0.1)
            v.mul_(0.999).add_(g * g, alpha=0.001)
            q -= 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"losses": torch.tensor(losses, dtype=torch.float64),
            "weights": torch.cat([q.reshape(-1) for q in P])}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("smooth", "filter"):
        return _smoothed(_mesh_params(case), _fields(case["fields"], case["nx"] * case["ny"] * case["nz"], seed))
    if kind in ("train", "infer"):
        w, x, t = _net(case, seed)
        return _network(case, w, x, t, case["steps"] if kind == "train" else 0)
    if kind not in ("average", "forces"):
        return None  # a trajectory: the state before the pass is the library's own
    L, parts = _bed(case, seed)
    p = _params(case, L)
    U, DU = _flow(p["ncell"], p["hi"], seed)
    if kind == "forces":
        return _forces(p, parts, U, DU)
    nx, ny, nz = p["ncell"]
    x, v, d = (torch.from_numpy(parts[k]).to(DEV) for k in ("x", "v", "d"))
    k = [((x[:, a] - p["lo"][a]) * (n / (p["hi"][a] - p["lo"][a]))).floor().clamp(0, n - 1).long()
         for a, n in enumerate((nx, ny, nz))]
    cell = (k[2] * ny + k[1]) * nx + k[0]
    vc = math.prod((p["hi"][a] - p["lo"][a]) / n for a, n in enumerate((nx, ny, nz)))
    vf = math.pi / 6 * d ** 3 / vc
    f = _fluid_force(p, x, 0.5 * d, v, U, DU)
    phi = torch.stack([torch.zeros(nx * ny * nz, dtype=torch.float64, device=DEV).index_add_(0, cell, q)
                       for q in [vf] + [vf * v[:, a] for a in range(3)] + [-f[:, a] / vc for a in range(3)]])
    phi = _smoothed(p, phi)
    mom = phi[1:4] * (phi[0] / phi[0].clamp(min=1e-12))
    return {"eps": phi[0], "mom": mom.T.contiguous(), "f": phi[4:7].T.contiguous()}
