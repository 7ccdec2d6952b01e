"""Timed workloads of the collisional-PIC step.

Each case is a piece of work a user has the framework do through its Python
classes, start to end: set a slab up and advance it, resume one from a
checkpoint, step a batch of admitted slabs, advance one's own particles.
The sizes are those of the repository's workloads (the small 1D slab, the 2D
foil, the large 2D study, the batched ensemble and the served requests, the
K-edge sweep, the thermalization and 10 keV runs, the transport mode), cut in
steps, and for the largest one in cells, so that a pass stays below a second.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what the user's program holds before the call
    run(state)           one pass and its outputs
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    the outputs in 64 bits, where plain numpy gives them
"""
import math

import numpy as np
import torch

import paper_1704_01202_gb300 as pkg
import pic_inputs as P
from paper_1704_01202_gb300 import kedge

ENERGIES = ("ke_e", "ke_i", "e_ion", "e_phot", "e_inc", "e_trans", "e_ka_esc", "e_esc", "e_field", "e_back",
            "e_rt_num", "e_rt_pend")


def _slab(name, nx, ny, dx, ppc_e, ppc_i, steps, **kw):
    c = dict(name=name, kind="slab", nx=nx, ny=ny, dx_nm=dx, ppc_e=ppc_e, ppc_i=ppc_i, z_init=3, steps=steps,
             hv_eV=1800.0, intensity=5e17, bins=2, ipd=1, photons=0.3, thermalize=False, coarsen=0, particles=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest served request (ensemble's lower end), run alone: every
        # step is launches and the latency of a few dozen tiny cells
        _slab("request_smallest_1d", 64, 1, 3.1, 26, 6, 100, particles=True),
        # the small 1D slab of the parity tests and the thermalization run,
        # resumed from a checkpoint some fs in, its charge states mixed
        _slab("small_slab_1d", 128, 1, 2.0, 256, 64, 100, kind="resume", hv_eV=1700.0, intensity=1.36e17, particles=True),
        # the 10 keV case with forced thermalization and Stewart-Pyatt
        # lowering: odd sizes, relativistic electrons, the other options
        _slab("extreme_10kev_1d", 257, 1, 2.0, 123, 31, 100, hv_eV=10000.0, intensity=1e19, bins=3, ipd=2,
              thermalize=True, particles=True),
        # a served request late in its run: stripped ions, cells of ~800-1200
        # electrons (the staging of the large-cell tiers)
        _slab("ionized_request_1d", 700, 1, 2.0, 820, 102, 64, z_init=8),
        # the 64 x 64-cell subdomain of the precision study, read back whole
        _slab("study_patch_2d", 64, 64, 5.0, 80, 20, 60, particles=True),
        # a slice of the 2D foil, ragged in x
        _slab("foil_slice_2d", 509, 64, 5.0, 64, 16, 100, hv_eV=1600.0, intensity=1e17, photons=0.05),
        # the 2D foil at its full 2048 x 256 cells
        _slab("foil_2d", 2048, 256, 5.0, 64, 16, 32, hv_eV=1600.0, intensity=1e17, photons=0.05),
        # the large 2D study on a quarter of its cells: the state is far
        # beyond the caches, memory and the per-cell kernels are everything
        _slab("study_2d", 4096, 512, 5.0, 80, 20, 12),
        # the foil with radiation transport (rad cells of 8 x 8, beam plus 8
        # diffuse ordinates, CIP) in place of the photon march
        _slab("transport_2d", 512, 256, 5.0, 64, 16, 40, hv_eV=1600.0, intensity=1e17, photons=0.0, coarsen=8),
        # the K-edge sweep: 12 photon energies x 2 lowering models in one
        # batch, a rad step every step
        dict(name="kedge_batch", kind="batch", slabs=24, nx=250, ppc_e=64, ppc_i=16, steps=100, ensemble=0),
        # a tick of the request loop: unequal slabs (cells and particles per
        # cell log-uniform) admitted, stepped and read out
        dict(name="ensemble_batch", kind="batch", slabs=20, nx=2048, ppc_e=0, ppc_i=0, steps=100, ensemble=7),
        # the user's own particles, push and fields alone (the process
        # switches of a collisionless run), read back whole
        dict(name="collisionless_2d", kind="loaded", nx=96, ny=48, dx_nm=5.0, ppc_e=32, ppc_i=8, steps=40),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["slab1", "slab1", "slab2", "slab2", "resume", "batch", "loaded"])
    hv = round(rng.uniform(1580.0, 1900.0), 1)
    inten = float("%.3g" % math.exp(rng.uniform(math.log(1e16), math.log(1e18))))
    if kind in ("slab1", "resume"):
        ppc = _log(rng, 32, 900)
        ppc_i = max(1, ppc // 5)
        nx = _log(rng, 64, max(65, min(4096, 1_500_000 // ppc)))
        c = _slab("", nx, 1, round(rng.uniform(1.0, 4.0), 2), ppc - ppc_i, ppc_i, rng.randint(24, 120), hv_eV=hv,
                  intensity=inten, bins=rng.randint(1, 4), ipd=rng.choice([1, 2]), thermalize=rng.random() < 0.2,
                  photons=round(rng.uniform(0.02, 0.5), 3), z_init=rng.choice([3, 3, 5, 8]),
                  particles=nx * ppc < 200_000)
        if kind == "resume":
            c.update(kind="resume", particles=True, steps=rng.randint(60, 150), nx=min(c["nx"], 1 + 150_000 // ppc))
    elif kind == "slab2":
        ppc = rng.randint(40, 160)
        ppc_i = ppc // 5
        n = _log(rng, 200_000, 20_000_000)
        nx = 8 * max(8, _log(rng, 64, 1024) // 8)
        ny = 8 * max(1, n // (ppc * nx * 8))
        c = _slab("", nx, ny, round(rng.uniform(4.0, 6.7), 2), ppc - ppc_i, ppc_i, rng.randint(16, 40), hv_eV=hv,
                  intensity=inten, photons=round(rng.uniform(0.02, 0.5), 3))
        if rng.random() < 0.25:
            c.update(coarsen=8, photons=0.0)
        elif rng.random() < 0.5:
            c.update(nx=nx + rng.randint(1, 7), ny=ny + rng.randint(1, 7))
    elif kind == "batch":
        if rng.random() < 0.5:
            c = dict(kind="batch", slabs=2 * rng.randint(4, 16), nx=rng.randint(100, 400), ppc_e=4 * rng.randint(8, 32),
                     ppc_i=rng.randint(8, 32), steps=rng.randint(32, 100), ensemble=0)
        else:
            c = dict(kind="batch", slabs=rng.randint(4, 20), nx=_log(rng, 256, 2048), ppc_e=0, ppc_i=0,
                     steps=rng.randint(32, 100), ensemble=rng.randint(1, 1000))
    else:
        c = dict(kind="loaded", nx=rng.randint(32, 128), ny=rng.randint(8, 48), dx_nm=5.0, ppc_e=4 * rng.randint(4, 10),
                 ppc_i=rng.randint(4, 10), steps=rng.randint(16, 40))
    c.pop("name", None)
    return c


def _members(c, seed):
    """(config, pulse) of every slab of a batch case."""
    if c["ensemble"]:
        m = P.batched_ensemble(c["slabs"], seed=c["ensemble"], cells=(64, c["nx"]))
        for k, (cfg, _) in enumerate(m):
            cfg.seed = 1000 * seed + k
        return m
    hv = np.linspace(1540.0, 1870.0, c["slabs"] // 2)
    return [(cfg, pl) for cfg, pl, _, _ in kedge.scan_slabs(P, hv, nx=c["nx"], ppc=(c["ppc_e"], c["ppc_i"]),
                                                            seed=1000 * seed)]


def _config(c, seed):
    flags = P.F_ALL | (P.F_THERM if c["thermalize"] else 0)
    return P.SlabConfig(nx=c["nx"], ny=c["ny"], dx_nm=c["dx_nm"], dy_nm=c["dx_nm"], ppc_e=c["ppc_e"],
                        ppc_i=c["ppc_i"], Z_init=c["z_init"], T_e_eV=100.0 if c["z_init"] == 8 else 10.0,
                        ipd_model=c["ipd"], seed=seed, flags=flags)


def prepare(c, seed):
    tables = P.standin_tables()
    s = dict(case=c, tables=tables)
    rng = np.random.default_rng(seed)
    if c["kind"] == "batch":
        # the server keeps its batch context; the requests' particles are host
        # arrays, as a client sends them
        s["members"] = [(cfg, P.init_particles(cfg), pl) for cfg, pl in _members(c, seed)]
        caps = [pkg.default_capacity(st.n_e, st.n_i, cfg.Z_init) for cfg, st, _ in s["members"]]
        s["rooms"] = sum(e for e, _ in caps), sum(i for _, i in caps)
        s["batch"] = pkg.Batch(tables, len(caps), max(cfg.nx for cfg, _, _ in s["members"]), *s["rooms"])
        return s
    if c["kind"] == "loaded":
        s["cfg"] = P.SlabConfig(nx=c["nx"], ny=c["ny"], dx_nm=c["dx_nm"], dy_nm=c["dx_nm"], ppc_e=c["ppc_e"],
                                ppc_i=c["ppc_i"], seed=seed, flags=P.F_PUSH | P.F_FIELD)
        s["particles"] = P.init_particles(s["cfg"])
        s["fields"] = P.random_fields(s["cfg"], seed + 1)
        return s
    s["cfg"] = cfg = _config(c, seed)
    s["rooms"] = pkg.default_capacity(cfg.ncell * cfg.ppc_e, cfg.ncell * cfg.ppc_i, cfg.Z_init) if c["particles"] else None
    # a pulse whose peak lies within the run's real horizon, seen on its rise
    s["pulse"] = P.Pulse(I_peak_Wcm2=c["intensity"], fwhm_fs=80.0, t_peak_fs=40.0, hv_eV=c["hv_eV"], n_bins=c["bins"])
    if c["photons"]:
        # the photon field of a slab the pulse already runs through
        s["photons"] = c["photons"] / c["bins"] * rng.uniform(0.5, 1.0, (cfg.ny, cfg.nx, c["bins"]))
    if c["kind"] == "resume":
        # the handle and the image of a run some fs in: charge states mixed
        slab = s["slab"] = pkg.Slab(cfg, tables, s["pulse"])
        slab.seed()
        slab.set_photons(s["photons"])
        slab.step(200)
        s["image"] = slab.checkpoint()
    return s


def _by_id(d, room):
    """Particles in the order of their ids (the library gives them cell by
    cell, in no order inside a cell), in the program's own arrays on the GPU,
    which have room for `room` of them."""
    ids = torch.from_numpy(d["id"].astype(np.int64)).cuda()
    order = torch.argsort(ids)
    if "slab" in d:                          # one order over all slabs of a batch: by slab, then id
        order = order[torch.argsort(torch.from_numpy(d["slab"]).cuda()[order], stable=True)]
    out = {}
    for k, v in d.items():
        v = ids if k == "id" else torch.from_numpy(v).cuda()
        out[k] = torch.zeros((room, *v.shape[1:]), dtype=v.dtype, device="cuda")
        torch.index_select(v, 0, order, out=out[k][:v.shape[0]])
    return out


def _diagnostics(slab, *slot):
    # the sums run over atomics in no fixed order, so they repeat to single
    # precision only; counts are whole numbers
    d = slab.diagnostics(*slot)
    return {"csd": d["csd"].astype(np.float32), "eedf": d["eedf"].astype(np.float32),
            "energies": np.array([d[k] for k in ENERGIES], dtype=np.float32),
            "plasma": np.array([d["T_e_eV"], d["Zbar"]], dtype=np.float32),
            "counts": np.array(list(d["counts"].values()) + [d["n_e"], d["n_i"]], dtype=np.int64)}


def _read(slab, rooms, photons):
    """What a user's program reads back at an output time: the grid fields, and
    the particles where they are few enough to be looked at one by one."""
    f = slab.fields()
    out = {"fields": np.stack([f[k] for k in ("ex", "ey", "ez", "bx", "by", "bz")]), "current": slab.current()}
    if photons:
        out["photons"] = slab.photons()
    if rooms:
        out["electrons"], out["ions"] = _by_id(slab.electrons(), rooms[0]), _by_id(slab.ions(), rooms[1])
    return out


def run(s):
    c = s["case"]
    if c["kind"] == "batch":
        b = s["batch"]
        slots = [b.admit(cfg, st, pl) for cfg, st, pl in s["members"]]
        b.step(c["steps"])
        rows = [_diagnostics(b, k) for k in slots]
        out = {k: np.stack([r[k] for r in rows]) for k in rows[0]}
        for species, get, room in (("electrons", b.electrons, s["rooms"][0]), ("ions", b.ions, s["rooms"][1])):
            parts = [get(k) for k in slots]
            for j, p in enumerate(parts):
                p["slab"] = np.full(p["id"].size, j, dtype=np.int32)
            out[species] = _by_id({k: np.concatenate([p[k] for p in parts]) for k in parts[0]}, room)
        for k in slots:
            b.retire(k)
        return out
    if c["kind"] == "resume":
        slab = s["slab"]
        slab.restore(s["image"])
        slab.step(c["steps"])
        return {**_diagnostics(slab), **_read(slab, s["rooms"], True)}
    if c["kind"] == "loaded":
        slab = pkg.Slab(s["cfg"], s["tables"])
        slab.load(s["particles"])
        slab.set_fields(s["fields"])
        slab.step(c["steps"])
        out = _read(slab, (s["particles"].n_e, s["particles"].n_i), False)
        slab.close()
        return out
    slab = pkg.Slab(s["cfg"], s["tables"], s["pulse"])
    if c["coarsen"]:
        slab.set_rt(coarsen=c["coarsen"], n_polar=4, n_azimuth=2, scheme=0)
    slab.seed()
    if "photons" in s:
        slab.set_photons(s["photons"])
    slab.step(c["steps"])
    out = {**_diagnostics(slab), **_read(slab, s["rooms"], True)}
    if c["coarsen"]:
        out["rt_field"] = slab.rt_field()[0]
    slab.close()
    return out


def work(c):
    """One read and one write of the 32 B particle record per step, the
    step's own minimum (nothing else of a step is of that size); about 400
    operations per collided particle and step, 150 for push and deposit."""
    if c["kind"] == "batch":
        n = sum(cfg.ncell * (cfg.ppc_e + cfg.ppc_i) for cfg, _ in _members(c, 0))
    else:
        n = c["nx"] * c["ny"] * (c["ppc_e"] + c["ppc_i"])
    return {"bytes": 64.0 * n * c["steps"], "flops": (150.0 if c["kind"] == "loaded" else 400.0) * n * c["steps"]}


# ---- 64-bit restatement of push, deposit and fields (2D, short moves) ----
_ME, _C, _QE, _EPS0 = 9.1093837015e-31, 299792458.0, 1.602176634e-19, 8.8541878128e-12
_C_NM_FS = 299.792458


def _shape4(x):
    """Linear weights at the nodes -1, 0, 1, 2."""
    return [np.maximum(0.0, 1.0 - np.abs(x - a)) for a in (-1, 0, 1, 2)]


def _gather(f, half_x, half_y, cx, cy, xi, eta):
    ny, nx = f.shape[0], f.shape[1] - 1
    xs, ys = xi - 0.5 * half_x, eta - 0.5 * half_y
    ax, ay = np.floor(xs).astype(int), np.floor(ys).astype(int)
    wx, wy = xs - ax, ys - ay
    out = np.zeros_like(xi)
    for a in (0, 1):
        i = cx + ax + a
        ok = (i >= 0) & (i <= (nx - 1 if half_x else nx))
        w = np.where(ok, wx if a else 1.0 - wx, 0.0)
        i = np.clip(i, 0, nx)
        for b in (0, 1):
            out += w * (wy if b else 1.0 - wy) * f[(cy + ay + b) % ny, i]
    return out


def _smooth(j, n):
    """(1/4, 1/2, 1/4) along x over the component's first n points, nothing
    beyond, and along y, periodic."""
    x = j[:, :n]
    sx = 0.5 * x
    sx[:, 1:] += 0.25 * x[:, :-1]
    sx[:, :-1] += 0.25 * x[:, 1:]
    out = np.zeros_like(j)
    out[:, :n] = 0.5 * sx + 0.25 * (np.roll(sx, 1, 0) + np.roll(sx, -1, 0))
    return out


def exact(c, seed):
    """Only the collisionless runs have a value without the framework's Monte
    Carlo method (its draws decide whole events)."""
    if c["kind"] != "loaded" or c["nx"] * c["ny"] * (c["ppc_e"] + c["ppc_i"]) * c["steps"] > 10_000_000:
        return None
    s = prepare(c, seed)
    cfg, p = s["cfg"], s["particles"]
    nx, ny, dx, dt = cfg.nx, cfg.ny, cfg.dx_nm, cfg.dt_fs
    W = nx + 1
    ex, ey, ez, bx, by, bz = (np.array(s["fields"][k], dtype=np.float64) for k in ("ex", "ey", "ez", "bx", "by", "bz"))
    E0 = _ME * _C / (_QE * 1e-15)
    kappa = _QE * cfg.n_ref_cm3 * 1e6 * 1e-9 / (_EPS0 * E0)
    cf = min(_C_NM_FS, cfg.cfl / (dt * math.sqrt(2.0 / dx ** 2)))
    mur = (cf * dt - dx) / (cf * dt + dx)
    sp = []
    for X, Y, u, q, w, m in ((p.eX, p.eY, p.eu, np.full(p.n_e, -1.0), p.ew.astype(np.float32), 1.0),
                             (p.iX, p.iY, p.iu, p.iZ + p.izf, np.full(p.n_i, cfg.w_ion), cfg.m_ion_me)):
        sp.append(dict(X=np.array(X), Y=np.array(Y), u=np.array(u, dtype=np.float64), q=q, w=np.array(w, dtype=np.float64),
                       m=m, live=np.ones(len(X), dtype=bool)))
    for _ in range(c["steps"]):
        J = np.zeros((3, ny * W))
        for d in sp:
            k = np.flatnonzero(d["live"])
            X, Y, u, q, w = d["X"][k], d["Y"][k], d["u"][k], d["q"][k], d["w"][k]
            cx, cy = np.floor(X).astype(int), np.floor(Y).astype(int)
            xi, eta = X - cx, Y - cy
            at = lambda f, hx, hy: _gather(f, hx, hy, cx, cy, xi, eta)  # noqa: E731
            e = np.stack([at(ex, 1, 0), at(ey, 0, 1), at(ez, 0, 0)], 1)
            b = np.stack([at(bx, 0, 1), at(by, 1, 0), at(bz, 1, 1)], 1)
            h = (0.5 * dt * q / d["m"])[:, None]
            um = u + h * e
            t = h * b / np.sqrt(1.0 + (um * um).sum(1))[:, None]
            up = um + np.cross(um, t)
            u = um + np.cross(up, t) * (2.0 / (1.0 + (t * t).sum(1)))[:, None] + h * e
            v = u / np.sqrt(1.0 + (u * u).sum(1))[:, None]
            x1, y1 = xi + v[:, 0] * _C_NM_FS * dt / dx, eta + v[:, 1] * _C_NM_FS * dt / dx
            if max(np.abs(x1 - xi).max(), np.abs(y1 - eta).max()) >= 1.0:
                return None
            qw = q * w
            S0x, S1x, S0y, S1y = _shape4(xi), _shape4(x1), _shape4(eta), _shape4(y1)
            put = lambda comp, a, bb, val: np.add(J[comp], np.bincount(  # noqa: E731
                ((cy + bb - 1) % ny) * W + np.clip(cx + a - 1, 0, nx),
                weights=np.where((cx + a - 1 >= 0) & (cx + a - 1 <= (nx - 1 if comp == 0 else nx)), val, 0.0),
                minlength=ny * W), out=J[comp])
            for bb in range(4):
                acc, sy = 0.0, 0.5 * (S0y[bb] + S1y[bb])
                for a in range(3):
                    acc = acc + (S1x[a] - S0x[a]) * sy
                    put(0, a, bb, -qw * acc)
            for a in range(4):
                acc, sx = 0.0, 0.5 * (S0x[a] + S1x[a])
                for bb in range(3):
                    acc = acc + (S1y[bb] - S0y[bb]) * sx
                    put(1, a, bb, -qw * acc)
                for bb in range(4):
                    dsx, dsy = S1x[a] - S0x[a], S1y[bb] - S0y[bb]
                    put(2, a, bb, qw * v[:, 2] * (S0x[a] * S0y[bb] + 0.5 * dsx * S0y[bb] + 0.5 * S0x[a] * dsy + dsx * dsy / 3.0))
            d["X"][k], d["Y"][k], d["u"][k] = cx + x1, (cy + y1) % ny, u
            d["live"][k[(d["X"][k] < 0) | (d["X"][k] >= nx)]] = False
        j3 = J.reshape(3, ny, W) * np.array([dx / dt, dx / dt, _C_NM_FS])[:, None, None]

        def b_half():
            hh = 0.5 * dt * cf / dx
            up_ = lambda f: np.roll(f, -1, 0)  # noqa: E731
            bx[:] -= hh * (up_(ez) - ez)
            by[:, :nx] += hh * (ez[:, 1:] - ez[:, :-1])
            bz[:, :nx] -= hh * ((ey[:, 1:] - ey[:, :-1]) - (up_(ex) - ex)[:, :nx])

        b_half()
        jx, jy, jz = _smooth(j3[0], nx), _smooth(j3[1], W), _smooth(j3[2], W)
        dn = lambda f: np.roll(f, 1, 0)  # noqa: E731
        nex, ney, nez = ex.copy(), ey.copy(), ez.copy()
        nex[:, :nx] += dt * (cf * (bz - dn(bz)) / dx - kappa * jx)[:, :nx]
        ney[:, 1:nx] += dt * (-cf * (bz[:, 1:nx] - bz[:, :nx - 1]) / dx - kappa * jy[:, 1:nx])
        nez[:, 1:nx] += dt * (cf * ((by[:, 1:nx] - by[:, :nx - 1]) - (bx - dn(bx))[:, 1:nx]) / dx - kappa * jz[:, 1:nx])
        for new, old in ((ney, ey), (nez, ez)):
            new[:, 0] = old[:, 1] + mur * (new[:, 1] - old[:, 0])
            new[:, nx] = old[:, nx - 1] + mur * (new[:, nx - 1] - old[:, nx])
        ex, ey, ez = nex, ney, nez
        b_half()
    out = {"fields": np.stack([ex, ey, ez, bx, by, bz]), "current": j3}
    for name, d, ids in (("electrons", sp[0], p.eid), ("ions", sp[1], p.iid)):
        k = np.flatnonzero(d["live"])
        k = k[np.argsort(ids[k])]
        room = lambda v: np.concatenate([v[k], np.zeros((len(v) - len(k), *v.shape[1:]))])  # noqa: E731
        out[name] = {"X": room(d["X"]), "Y": room(d["Y"]), "u": room(d["u"]), "id": None}
        if name == "electrons":
            out[name]["w"] = room(d["w"])
        else:
            out[name].update(zf=room(p.izf), Z=None, nK=None)
    return out
