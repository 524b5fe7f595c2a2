"""The workloads this library is measured on: whole calls a user's program makes.

Every pass is one piece of a run through the public entry points (the
`Simulation` class of `lbm.py`, or the C ABI it binds): the initial condition
from host arrays, `steps` time steps, and the read-back the program does at
that point.  Each pass starts again from its own initial phase field, so all
passes on one state do the same work.

A case is plain numbers:

  kind       "drop" (static drop), "p2" (oscillating drop), "ellipsoid", "thread",
             "bubble": one grid of nz x nr nodes; "sweep": `ncases` drops on the
             grids of `workloads.batched_cases`, advanced as one batch
  precision  storage form of `lbm_params` (fp64, fp32, mix_fp16, mix_bf16)
  z_periodic, lagged, raw, bgk
             periodic z; lagged pressure coupling; raw-moment collision; all
             rates equal (the general-rate kernels)
  steps      time steps between two readings
  read       what is read then: "monitor" (the diagnostics record alone), "record"
             (the record and the fields), "fields" (phi, rho, u, p), "drops" (the
             axis drops, phi and u), "phi"
             (phi of every case of a sweep, into one pinned host buffer),
             "resume" (a stored state is set, stepped and read back)
"""
import ctypes
import math

import numpy as np
import torch

from paper_1810_09299_gb300 import lbm, workloads

RECORD = ("step", "mass", "kinetic", "z_centroid", "dp", "umax", "phi_min", "phi_max", "axis_half_length",
          "radial_half_length", "nonfinite")
FIELDS = ("phi", "rho", "uz", "ur", "p")
STATE_BYTES = {"fp64": 160, "fp32": 84, "mix_fp16": 46, "mix_bf16": 50}  # f, g, chi of one node, stored once
FLOPS_PER_NODE = 400  # one node update of Eq. 16-40, counted in adds and multiplies


def _one(name, kind, nr, nz, precision, steps, read, **kw):
    c = dict(name=name, kind=kind, nr=nr, nz=nz, precision=precision, steps=steps, read=read, ncases=1,
             z_periodic=0, lagged=0, raw=0, bgk=0)
    c.update(kw)
    return c


def listed():
    return [
        # a monitoring loop on the smallest drop: one step, one record (C ABI default precision)
        _one("monitor_64x128_fp64", "drop", 64, 128, "fp64", 1, "monitor"),
        # the static drop of Sec. 3.1, advanced between two readings
        _one("drop_64x128_fp64", "drop", 64, 128, "fp64", 100, "fields"),
        # the oscillating drop of Sec. 3.2, polled for its axis lengths
        _one("p2_128x256_fp64", "p2", 128, 256, "fp64", 40, "record"),
        _one("p2_128x256_fp32", "p2", 128, 256, "fp32", 400, "record"),
        # the liquid thread of Sec. 3.3 in 16-bit storage, polled for its breakup
        _one("thread_64x180_fp16", "thread", 64, 180, "mix_fp16", 500, "drops", z_periodic=1),
        # the paper's own thread (its grid and density scale), polled every 40 steps
        _one("thread_200x600_fp64", "thread", 200, 600, "fp64", 40, "drops", z_periodic=1, paper=1),
        # the rising bubble at full size
        _one("bubble_256x1024_fp32", "bubble", 256, 1024, "fp32", 200, "fields"),
        # the raw-moment collision on a ragged grid in bfloat16 storage
        _one("raw_101x333_bf16", "p2", 101, 333, "mix_bf16", 300, "fields", raw=1),
        # a parameter sweep of 512 drops: the benchmark's batch, in both of its forms
        _one("sweep_512_fp32", "sweep", 0, 0, "fp32", 128, "phi", ncases=512),
        _one("sweep_512_fp16", "sweep", 0, 0, "mix_fp16", 128, "phi", ncases=512),
        # a sweep in full precision
        _one("sweep_64_fp64", "sweep", 0, 0, "fp64", 10, "phi", ncases=64),
        # a stored state set again, advanced and read back (resuming a run)
        _one("resume_150x300_fp32", "ellipsoid", 150, 300, "fp32", 100, "resume", z_periodic=1, paper=1),
    ]


def draw(rng):
    prec = rng.choice(["fp64", "fp64", "fp32", "fp32", "mix_fp16", "mix_bf16"])
    kind = rng.choice(["drop", "p2", "ellipsoid", "thread", "bubble", "sweep"])
    if kind == "sweep":
        n = int(round(math.exp(rng.uniform(math.log(3), math.log(200)))))
        steps = rng.randint(3, 12) if prec == "fp64" else rng.randint(20, 100)
        return _strip(_one("", "sweep", 0, 0, prec, steps, "phi", ncases=n, raw=int(prec != "fp64" and rng.random() < 0.3)))
    nr = int(round(math.exp(rng.uniform(math.log(32), math.log(300)))))
    nz = int(round(nr * rng.uniform(1.6, 4.0)))
    raw = int(rng.random() < 0.2)
    bgk = int(not raw and rng.random() < 0.15)
    # FP64: inside the horizon over which runs that round differently stay together (inside a large
    # drop phi = 1 and the interface normal's direction is round-off; it grows after 20-30 steps)
    if prec == "fp64":
        steps = rng.randint(1, 30) if kind == "thread" and not raw else rng.randint(1, 12)
    else:
        steps = int(round(math.exp(rng.uniform(math.log(4), math.log(400)))))
    return _strip(_one("", kind, nr, nz, prec, steps, rng.choice(["monitor", "record", "fields", "drops", "resume"]), raw=raw, bgk=bgk,
                       z_periodic=int(kind == "thread" or rng.random() < 0.3), lagged=int(rng.random() < 0.15)))


def _strip(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------- inputs
def _params(case, seed):
    """The case dicts of workloads.py, their shapes jittered by the seed."""
    rng = np.random.default_rng(seed)
    nr, nz, kind, prec = case["nr"], case["nz"], case["kind"], case["precision"]
    if kind == "sweep":
        out = workloads.batched_cases(case["ncases"], precision=prec)  # the benchmark's grids and drops
        for c in out:
            c["shape_args"][0] += float(rng.uniform(-2.0, 2.0))
            c["shape_args"][1] *= float(rng.uniform(0.95, 1.0))
    else:
        j = lambda a, b: float(rng.uniform(a, b))  # noqa: E731
        zc = nz * j(0.48, 0.52)
        if kind == "drop":
            c = workloads.static_drop(nr=nr, nz=nz, R=nr * j(0.24, 0.26), zc=zc)
        elif kind == "p2":
            c = workloads.oscillating_drop(nr=nr, nz=nz, R0=nr * j(0.24, 0.26), eps=j(0.03, 0.07), zc=zc)
        elif kind == "ellipsoid":
            c = workloads.paper_ellipsoid(Rr=0.2 * nr * j(0.9, 1.1), Rz=0.3 * nz * j(0.9, 1.1))
            c.update(nr=nr, nz=nz)
            c["shape_args"][0] = zc
        elif kind == "thread":
            c = workloads.paper_thread() if case.get("paper") else workloads.thread_breakup(nr=nr)
            R = 0.3 * nr * j(0.95, 1.05)
            c.update(nr=nr, nz=nz, shape_args=[R, 0.1 * R, float(nz), j(0.0, 6.28), 4.0])
        else:
            R = nr * j(0.12, 0.16)
            c = workloads.rising_bubble(nr=nr, nz=nz, R=R, zc=nz * j(0.2, 0.3))
            c["grav_z"] *= (R / 32.0) ** 2
        c["z_periodic"] = case["z_periodic"]
        out = [c]
    for i, c in enumerate(out):
        if case["raw"]:
            out[i] = c = workloads.with_raw_collision(c)
        if case["bgk"]:
            c.update(sf=[-1.0] * 9, sg=[-1.0] * 9)
        c.update(precision=prec, p_coupling=case["lagged"])
    return out


def _phi0(c, dev):
    """The initial phase field of a case dict ([nz, nr] doubles on `dev`)."""
    z = torch.arange(c["nz"], dtype=torch.float64, device=dev)[:, None] + 0.5
    r = torch.arange(c["nr"], dtype=torch.float64, device=dev)[None, :] + 0.5
    a, s = c["shape_args"], c["shape"]
    if s == "thread":
        x = a[0] + a[1] * torch.cos(2.0 * math.pi * z / a[2] + a[3]) - r
    else:
        d = torch.sqrt((z - a[0]) ** 2 + r ** 2)
        if s == "p2":
            x = a[1] * (1.0 + a[2] * 0.5 * (3.0 * ((z - a[0]) / d) ** 2 - 1.0)) - d
        elif s == "ellipsoid":
            q = torch.sqrt((z - a[0]) ** 2 / a[1] ** 2 + r ** 2 / a[2] ** 2)
            x = (a[2] * a[2] * a[1]) ** (1.0 / 3.0) * (1.0 - q)
        else:
            x = a[1] - d
    v = 0.5 + 0.5 * torch.tanh(2.0 * x / c["W"])
    return 1.0 - v if s == "bubble" else v


def _resting_state(c, phi0):
    """f, g and (chi, p) of the resting state of phi0: what a stored state holds at its start."""
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    cr = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]
    r = np.arange(c["nr"])[None, None, :] + 0.5
    f = np.ascontiguousarray(w * phi0[None] * (r + 3.0 * c["mobility"] * cr))
    aux = np.zeros((3,) + phi0.shape)
    aux[1] = c["mobility"] * phi0
    return f, np.zeros_like(f), aux


def prepare(case, seed):
    cs = _params(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    sizes = [c["nz"] * c["nr"] for c in cs]
    pin = dev == "cuda"
    phi = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=pin)
    o = 0
    for c, n in zip(cs, sizes):
        phi[o:o + n].copy_(_phi0(c, dev).reshape(-1), non_blocking=pin)
        o += n
    if pin:
        torch.cuda.synchronize()
    s = {"case": dict(case), "phi": phi, "sim": lbm.Simulation(cs)}
    if case["kind"] == "sweep":
        s["offsets"] = [0] + np.cumsum(sizes).tolist()
        s["out"] = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=pin)
        # long runs pick their launch shape once, on their own state
        s["sim"].init_all(phi.numpy())
        s["sim"].autotune()
    elif case["read"] == "resume":
        s["stored"] = _resting_state(cs[0], phi.numpy().reshape(cs[0]["nz"], cs[0]["nr"]))
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    case, sim = state["case"], state["sim"]
    phi = state["phi"].numpy()
    if case["kind"] == "sweep":
        sim.init_all(phi)
        sim.step(case["steps"])
        lib, out, off = lbm.lib(), state["out"], state["offsets"]
        dp = ctypes.POINTER(ctypes.c_double)
        for c in range(case["ncases"]):
            rc = lib.lbm_case_get_fields(sim.handle, c, 1, ctypes.cast(out.data_ptr() + 8 * off[c], dp))
            if rc != lbm.LBM_OK:
                raise lbm.LbmError(rc, "lbm_case_get_fields")
        return {"phi": out}
    if case["read"] == "resume":
        sim.set_state(0, *state["stored"])
        sim.step(case["steps"])
        f, g, aux = sim.state(0)
        return {"f": f, "g": g, "aux": aux}
    sim.init_phase(0, "host_array", phi=phi.reshape(sim.cases[0]["nz"], sim.cases[0]["nr"]))
    sim.step(case["steps"])
    if case["read"] == "drops":
        drops, n, (phi_min, z_min) = sim.axis_drops(0)
        out = sim.fields(0, ("phi", "uz", "ur"))
        out["drops"] = np.array([n, phi_min] + [d[k] for d in drops for k in ("volume", "radius")])
        return out
    out = {}
    if case["read"] in ("monitor", "record"):
        record = sim.diagnostics(0)
        out["record"] = np.array([record[k] for k in RECORD])
    if case["read"] != "monitor":
        out.update(sim.fields(0))
    return out


def _nodes(case):
    if case["kind"] != "sweep":
        return case["nr"] * case["nz"]
    return sum(c["nr"] * c["nz"] for c in workloads.batched_cases(case["ncases"]))


def work(case):
    # every step reads and writes the state once; the read-back writes FP64 values
    n = _nodes(case)
    values = {"monitor": 0, "record": 5, "fields": 5, "drops": 3, "phi": 1, "resume": 42}[case["read"]]
    return {"bytes": n * (2.0 * STATE_BYTES[case["precision"]] * case["steps"] + 8.0 * (values + 1)),
            "flops": float(FLOPS_PER_NODE) * n * case["steps"]}


# ---------------------------------------------------------------- the same in 64 bits
CZ = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CR = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
RMIR = (0, 1, 4, 3, 2, 8, 7, 6, 5)
M = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
              CZ, [0, -2, 0, 2, 0, 1, -1, -1, 1], CR, [0, 0, -2, 0, 2, 1, 1, -1, -1],
              [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)
_cz, _cr = np.array(CZ, float), np.array(CR, float)
RAW = np.array([_cz * 0 + 1, _cz, _cr, _cz**2 + _cr**2, _cz**2 - _cr**2, _cz * _cr, _cz**2 * _cr, _cz * _cr**2,
                _cz**2 * _cr**2])


class _Flat:
    """Every node of every grid in one flat array, with its neighbours' places."""

    def __init__(self, cs, dev):
        self.cs, self.n = cs, sum(c["nz"] * c["nr"] for c in cs)
        self.dev = dev
        ten = lambda: torch.empty(self.n, dtype=torch.float64, device=dev)  # noqa: E731
        self.r, self.par = ten(), {}
        self.near = {}  # (dz, dr) -> place of the node there, mirrored or wrapped
        offs = [(a * CZ[i], a * CR[i]) for a in (1, 2) for i in range(1, 9)]
        for d in offs:
            self.near[d] = torch.empty(self.n, dtype=torch.int64, device=dev)
        self.src = [None] + [torch.empty(self.n, dtype=torch.int64, device=dev) for _ in range(8)]
        same = lambda k: all(c[k] == cs[0][k] for c in cs)  # noqa: E731
        for k in ("rho_l", "rho_g", "nu_l", "nu_g", "sigma", "W", "mobility", "grav_z", "n_eps"):
            self.par[k] = cs[0][k] if same(k) else ten()
        o = 0
        for c in cs:
            nz, nr, per = c["nz"], c["nr"], c["z_periodic"]
            m = nz * nr
            k = torch.arange(nz, device=dev)[:, None].expand(nz, nr)
            j = torch.arange(nr, device=dev)[None, :].expand(nz, nr)
            self.r[o:o + m] = (j + 0.5).reshape(-1).double()
            for key, v in self.par.items():
                if torch.is_tensor(v):
                    v[o:o + m] = c[key]

            def ghost(kk, jj):
                jj = torch.where(jj < 0, -1 - jj, torch.where(jj >= nr, 2 * nr - 1 - jj, jj))
                kk = kk % nz if per else torch.where(kk < 0, -1 - kk, torch.where(kk >= nz, 2 * nz - 1 - kk, kk))
                return (o + kk * nr + jj).reshape(-1)

            for d in offs:
                self.near[d][o:o + m] = ghost(k + d[0], j + d[1])
            for i in range(1, 9):  # where the population arriving along c_i was
                ks, js = k - CZ[i], j - CR[i]
                if per:
                    ks, zout = ks % nz, torch.zeros_like(ks, dtype=torch.bool)
                else:
                    zout = (ks < 0) | (ks >= nz)
                back = zout | (js >= nr)
                axis = (js < 0) & ~back
                d = torch.where(back, OPP[i], torch.where(axis, RMIR[i], i))
                ks, js = torch.where(back, k, ks), torch.where(back, j, torch.where(axis, torch.zeros_like(js), js))
                self.src[i][o:o + m] = (d * self.n + o + ks * nr + js).reshape(-1)
            o += m

    def macros(self, f, g, p_prev):
        """phi, its stencils, and u and p, from the populations."""
        c, P, r = self.cs[0], self.par, self.r
        q = {"phi": f.sum(0) / r}
        phi = q["phi"]
        q["gz"], q["gr"], q["lap"] = torch.zeros_like(phi), torch.zeros_like(phi), torch.zeros_like(phi)
        for i in range(1, 9):
            x1, x2 = phi[self.near[(CZ[i], CR[i])]], phi[self.near[(2 * CZ[i], 2 * CR[i])]]
            d = (8.0 * x1 - x2) * (WT[i] / 2.0)
            if CZ[i]:
                q["gz"] += CZ[i] * d
            if CR[i]:
                q["gr"] += CR[i] * d
            q["lap"] += (16.0 * x1 - x2 - 15.0 * phi) * (WT[i] / 2.0)
        gz, gr, dr = q["gz"], q["gr"], P["rho_l"] - P["rho_g"]
        rho = q["rho"] = P["rho_g"] + phi * dr
        nu = q["nu"] = phi * P["nu_l"] + (1.0 - phi) * P["nu_g"]
        beta, kap = 12.0 * P["sigma"] / P["W"], 1.5 * P["sigma"] * P["W"]
        mu = 4.0 * beta * phi * (phi - 1.0) * (phi - 0.5) - kap * q["lap"] - kap * gr / r
        Fsz, Fsr, Gz = mu * gz, mu * gr, (rho - P["rho_l"]) * P["grav_z"]
        tau = 3.0 * nu + 0.5
        sg = q["sg"] = [1.0 / tau if s < 0 else s for s in c["sg"]]
        Jz, Jr = sum(CZ[i] * g[i] for i in range(9) if CZ[i]), sum(CR[i] * g[i] for i in range(9) if CR[i])
        S0 = g[1:].sum(0)
        if c["collision"]:
            sp = 1.5 / sg[3] - 0.5 / sg[8] - 0.5
        else:
            sp = (sg[1] + sg[2] - sg[1] * sg[2]) / (2.0 * sg[1] * sg[2])
        uz = (Jz + 0.5 * r * (Fsz + Gz)) / (r * rho)
        D = r * rho + nu * rho / r
        A0 = 0.6 * (S0 / r + 0.5 * uz * dr * gz - (2 / 3) * rho * uz * uz)
        A1 = 0.6 * (0.5 * dr * gr - sp * (4 / 9) * rho / r)
        A2 = 0.4 * rho
        if c["p_coupling"]:
            ps = p_prev
            ur = (Jr + 0.5 * (r * Fsr + ps)) / D
            p = A0 + A1 * ur - A2 * ur * ur
        else:
            a, b = (Jr + 0.5 * r * Fsr) / D, 0.5 / D
            qa, qb, qc = A2 * b * b, 1.0 - A1 * b + 2.0 * A2 * a * b, -(A0 + A1 * a - A2 * a * a)
            disc = qb * qb - 4.0 * qa * qc
            p = torch.where(disc >= 0, -2.0 * qc / (qb + torch.sqrt(disc.clamp(min=0.0))), -qc / qb)
            ps, ur = p, a + b * p
        q.update(uz=uz, ur=ur, p=p, Fz=r * (Fsz + Gz), Fr=r * Fsr + ps - 2.0 * rho * nu * ur / r)
        return q

    def collide(self, x, eq, src, rates):
        """x - B^-1 S B (x - eq) + B^-1 (1 - S/2) B src for moments `eq`, `src` of the orthogonal basis."""
        raw = self.cs[0]["collision"]
        dev, T = self.dev, lambda a: torch.tensor(a, dtype=torch.float64, device=self.dev)  # noqa: E731
        m = torch.matmul(T(M), x.reshape(9, -1))
        d, s = m - torch.stack(eq), torch.stack(src)
        if raw:
            A = T(RAW @ np.linalg.inv(M))
            d, s = A @ d, A @ s
        for i in range(9):
            d[i] = -rates[i] * d[i] + (1.0 - 0.5 * rates[i]) * s[i]
        return x + T(np.linalg.inv(RAW if raw else M)) @ d

    def step(self, f, g, chi, p_prev):
        c, P, r = self.cs[0], self.par, self.r
        q = self.macros(f, g, p_prev)
        phi, rho, uz, ur, p = (q[k] for k in FIELDS)
        gn = torch.sqrt(q["gz"] ** 2 + q["gr"] ** 2) + P["n_eps"]
        lam = 4.0 * phi * (1.0 - phi) / P["W"]
        cz, cr = r * phi * uz, r * phi * ur + P["mobility"] * phi
        R1, R2 = cz - chi[0] + r * lam * q["gz"] / gn / 3.0, cr - chi[1] + r * lam * q["gr"] / gn / 3.0
        o, rp = torch.zeros_like(phi), r * phi
        sf = [1.0 / (3.0 * P["mobility"] + 0.5) if s < 0 else s for s in c["sf"]]
        fp = self.collide(f, [rp, -2 * rp, rp, cz, -cz, cr, -cr, o, o], [o, o, o, R1, -R1, R2, -R2, o, o], sf)
        dr, u2 = P["rho_l"] - P["rho_g"], uz * uz + ur * ur
        a, b = r * dr * q["gz"], rho + r * dr * q["gr"]
        ud = uz * a + ur * b
        eq = [o, 3 * r * (2 * p + rho * u2), -3 * r * (3 * p + rho * u2), r * rho * uz, -r * rho * uz, r * rho * ur,
              -r * rho * ur, r * rho * (uz * uz - ur * ur), r * rho * ur * uz]
        T = [ud - rho * ur, 2 * rho * ur, -ud - rho * ur, q["Fz"], -q["Fz"], q["Fr"], -q["Fr"],
             (2 / 3) * (uz * a - ur * b), (uz * b + ur * a) / 3.0]
        gp = self.collide(g, eq, T, q["sg"])
        fn, gn = torch.empty_like(f), torch.empty_like(g)
        fn[0], gn[0] = fp[0], gp[0]
        for i in range(1, 9):
            fn[i], gn[i] = fp.reshape(-1)[self.src[i]], gp.reshape(-1)[self.src[i]]
        return fn, gn, (cz, cr), p


def _record(c, q, steps):
    """The diagnostics record of one case (the definitions of lbm_diag)."""
    nz, nr, per = c["nz"], c["nr"], c["z_periodic"]
    phi, rho, uz, ur, p = (q[k].reshape(nz, nr).cpu().numpy() for k in FIELDS)
    z, r = np.arange(nz)[:, None] + 0.5, np.arange(nr)[None, :] + 0.5
    mass, uu = (r * phi).sum(), uz * uz + ur * ur
    zc = (r * z * phi).sum() / mass
    mean = lambda m: (r * p)[m].sum() / (r + 0 * p)[m].sum() if m.any() else 0.0  # noqa: E731
    a = phi[:, 0] - 0.5
    length = 0.5 if not per and a[0] > 0 else 0.0
    for k in range(nz):
        if k + 1 == nz and not per:
            length += 0.5 if a[k] > 0 else 0.0
            continue
        x, y = a[k], a[(k + 1) % nz]
        length += 1.0 if x > 0 and y > 0 else x / (x - y) if x > 0 else y / (y - x) if y > 0 else 0.0
    row = phi[min(max(int(math.floor(zc)), 0), nz - 1)] - 0.5
    cross = [j for j in range(nr - 1) if row[j] > 0 and row[j + 1] <= 0]
    rad = cross[0] + 0.5 + row[cross[0]] / (row[cross[0]] - row[cross[0] + 1]) if cross else 0.0
    return dict(step=float(steps), mass=mass, kinetic=(0.5 * r * rho * uu).sum(), z_centroid=zc,
                dp=mean(phi > 0.99) - mean(phi < 0.01), umax=math.sqrt(uu.max()), phi_min=phi.min(), phi_max=phi.max(),
                axis_half_length=0.5 * length, radial_half_length=rad, nonfinite=0.0)


def exact(case, seed):
    n = _nodes(case)
    if n * case["steps"] > 4.5e9:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    cs = _params(case, seed)
    F = _Flat(cs, dev)
    phi = torch.cat([_phi0(c, dev).reshape(-1) for c in cs])
    mob = F.par["mobility"]
    f = torch.stack([WT[i] * phi * (F.r + 3.0 * CR[i] * mob) for i in range(9)])
    g = torch.zeros_like(f)
    chi, p = (torch.zeros_like(phi), mob * phi), torch.zeros_like(phi)
    for _ in range(case["steps"]):
        f, g, chi, p = F.step(f, g, chi, p)
    # velocities, g and chi of a slow flow in 16-bit storage carry that storage's rounding, not the method's value
    wide = not case["precision"].startswith("mix")
    if case["read"] == "resume":
        shape = (cs[0]["nz"], cs[0]["nr"])
        host = lambda x: x.reshape((-1,) + shape).cpu().numpy()  # noqa: E731
        # p^{n-1} is part of the state under the lagged coupling only
        aux = torch.stack([chi[0], chi[1], p if case["lagged"] else torch.zeros_like(p)])
        return {"f": host(f), "g": host(g) if wide else None, "aux": host(aux) if wide else None}
    if case["kind"] == "sweep":
        return {"phi": (f.sum(0) / F.r).cpu().numpy()}
    q = F.macros(f, g, p)
    c = cs[0]
    host = lambda k: q[k].reshape(c["nz"], c["nr"]).cpu().numpy() if wide or k not in ("uz", "ur") else None  # noqa: E731
    if case["read"] == "drops":
        out = {k: host(k) for k in ("phi", "uz", "ur")}
        axis, vol = out["phi"][:, 0], 2.0 * math.pi * float((F.r * q["phi"]).sum())
        whole = bool((axis > 0.5).all())  # an unbroken body; the cuts between drops have no 64-bit restatement here
        out["drops"] = np.array([1.0, axis.min(), vol, (3.0 * vol / (4.0 * math.pi)) ** (1.0 / 3.0)]) if whole else None
        return out
    out = {}
    if case["read"] in ("monitor", "record"):
        record = _record(c, q, case["steps"])
        out["record"] = np.array([record[k] for k in RECORD])
    if case["read"] != "monitor":
        out.update({k: host(k) for k in FIELDS})
    return out
