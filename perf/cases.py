"""What a user of this library has it do, as cases that can be timed and compared.

A case is one solver with its domains; a pass advances them by `steps` time
steps and reads the result back, as a program does between two snapshots or
checkpoints (eulbfs.Solver.step, then fields or save), or serves a handful of
requests from creation to the diagnostics of each (serving.serve).

The problems are those of `workloads`: conductive and three-phase Stefan
layers, a film under gravity, droplets on a cold plate (planar and of
revolution, with fixed and hysteresis contact angles), batches of uneven
droplet domains, a domain split into slabs.  FP32C results are read as raw
checkpoints (`save`: the state planes in single precision, H and C as hi/lo
pairs, with F_s of the previous step), FP64 results as fields or checkpoints.
A seed sets contact angles, Stefan numbers, density ratios, plate
temperatures and surface waves; sizes and steps belong to the case.

`exact` is the method in 64 bits, written with plain torch operations: every
surrounding point of every face, every equilibrium and every moment as a sum
over the nine directions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_03366_gb300 import eulbfs, serving, workloads as wl

PRECISION = {"fp64": eulbfs.FP64, "fp32c": eulbfs.FP32C}

# Bytes of a cell that a step has to read and write once (the state and F_s
# of the previous step), and floating-point operations of its three stages.
BYTES = {"fp64": 96, "fp32c": 64}
FLOPS = 3 * 905


def listed():
    return [
        # The smallest: the one-phase Stefan problem as a verification run in
        # FP64, four rows of 256 cells, profiles read every 16 steps.
        {"name": "stefan_256x4_fp64", "kind": "stefan", "nx": 256, "ny": 4, "precision": "fp64", "steps": 16},
        # Layers of solid, liquid and gas, the longest of the 1-D problems.
        {"name": "layers_1024x4", "kind": "layers", "nx": 1024, "ny": 4, "precision": "fp32c", "steps": 64},
        # One small droplet of revolution.
        {"name": "droplet_128_rz", "kind": "droplet", "nx": 128, "ny": 128, "axi": True, "precision": "fp32c",
         "steps": 64},
        # A planar droplet on a hysteresis plate, on the 400 x 200 grid of the droplet runs.
        {"name": "droplet_400x200", "kind": "droplet", "nx": 400, "ny": 200, "axi": False, "hysteresis": True,
         "precision": "fp32c", "steps": 200},
        # A ragged domain whose rows are not a multiple of 16 bytes.
        {"name": "film_333x251", "kind": "film", "nx": 333, "ny": 251, "precision": "fp32c", "steps": 100},
        # The film of the repository's test and benchmark size.
        {"name": "film_512", "kind": "film", "nx": 512, "ny": 512, "precision": "fp32c", "steps": 200},
        # One droplet in FP64, all its fields read: an accuracy run.
        {"name": "droplet_256_rz_fp64", "kind": "droplet", "nx": 256, "ny": 256, "axi": True, "precision": "fp64",
         "steps": 50},
        # A domain split into four slabs (halo copies between the stages).
        {"name": "split_768_in_4", "kind": "droplet", "nx": 768, "ny": 768, "axi": True, "slabs": 4,
         "precision": "fp32c", "steps": 60},
        # Six requests of freezing droplets on the hysteresis plate through the
        # serving loop, admission to diagnostics.
        {"name": "serve_6", "kind": "serve", "domains": 6, "lo": 256, "hi": 512, "axi": True, "precision": "fp32c",
         "steps": 96},
        # An ordinary batch with streaming steps below one half, planar.
        {"name": "batch_16_streaming", "kind": "batch", "domains": 16, "axi": False, "streaming": True,
         "precision": "fp32c", "steps": 50},
        # The plain FP64 step of a batch, for comparison and reference runs.
        {"name": "batch_16_fp64", "kind": "batch", "domains": 16, "axi": True, "precision": "fp64", "steps": 12},
        # The largest: the static-droplet batch of the benchmark, 64 uneven domains of revolution.
        {"name": "batch_64_rz", "kind": "batch", "domains": 64, "axi": True, "precision": "fp32c", "steps": 200},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same families: sizes over their whole range, odd
    ones among them, steps so that a pass costs less than the largest listed
    case's."""
    kind = rng.choice(["stefan", "layers", "film", "droplet", "droplet", "droplet", "batch", "batch", "serve"])
    precision = "fp64" if rng.random() < 0.25 else "fp32c"
    if kind in ("stefan", "layers"):
        case = {"kind": kind, "nx": _log_size(rng, 96, 2048), "ny": rng.randint(2, 9)}
    elif kind == "film":
        case = {"kind": kind, "nx": _log_size(rng, 96, 1024), "ny": _log_size(rng, 96, 1024)}
    elif kind == "droplet":
        case = {"kind": kind, "nx": _log_size(rng, 64, 1024), "ny": _log_size(rng, 64, 1024),
                "axi": rng.random() < 0.6, "hysteresis": rng.random() < 0.4}
        if precision == "fp32c" and rng.random() < 0.2:
            case["slabs"] = rng.randint(2, min(6, case["ny"] // 8))
        elif rng.random() < 0.2:
            case["streaming"] = True
    elif kind == "serve":
        case = {"kind": kind, "domains": rng.randint(2, 6), "lo": 128, "hi": 640, "axi": rng.random() < 0.5}
        precision = "fp32c"
    else:
        case = {"kind": kind, "domains": _log_size(rng, 4, 64), "axi": rng.random() < 0.6,
                "streaming": rng.random() < 0.3}
    case["precision"] = precision
    most = {"fp64": 2.0e7, "fp32c": 4.0e8}[precision]
    case["steps"] = max(4, min(rng.randint(12, 200), int(most / _cells(dict(case, steps=1)))))
    return case


# -- problems -----------------------------------------------------------------

def _sides(case):
    """Sides of a batch's or a serving trace's square domains (they belong to the case, not to the seed)."""
    rng = np.random.default_rng(1000 + case["domains"])
    if case["kind"] == "serve":
        return [int(round(rng.uniform(case["lo"], case["hi"]) / 32.0)) * 32 for _ in range(case["domains"])]
    return [int(s) for s in rng.choice(wl.BATCH_SIDES, size=case["domains"])]


def _cells(case):
    if case["kind"] in ("batch", "serve"):
        return sum(s * s for s in _sides(case))
    return case["nx"] * case["ny"]


def _droplet(rng, side, axi, hysteresis=False, streaming=False):
    theta = 82.0 if hysteresis else float(rng.uniform(60, 150))
    c = wl.droplet(side, theta_deg=theta, St=float(rng.uniform(0.05, 0.5)), rho_sl=float(rng.uniform(0.85, 0.95)),
                   Tw=float(rng.uniform(-1.0, -0.2)), axisymmetric=axi,
                   hysteresis=(100.0, 39.0) if hysteresis else None)
    if streaming:
        c.dt_h, c.dt_f, c.dt_g = 0.3, 0.4, 0.3
    return c


def _problems(case, seed):
    """The workloads.Case of every domain."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "stefan":
        return [wl.conductive(case["nx"], case["ny"], St=float(rng.uniform(0.1, 1.0)),
                              alpha=float(rng.uniform(0.05, 0.1)))]
    if kind == "layers":
        return [wl.three_phase(case["nx"], case["ny"], St=float(rng.uniform(0.1, 1.0)),
                               H0=case["nx"] * float(rng.uniform(0.1, 0.5)),
                               rho_ratio_sl=float(rng.uniform(0.85, 0.95)))]
    if kind == "film":
        n = max(case["nx"], case["ny"])
        return [wl.film(n, seed=seed, height=float(rng.uniform(0.2, 0.4)) * case["ny"] / n,
                        St=float(rng.uniform(0.1, 0.4))).crop(case["nx"], case["ny"])]
    if kind == "droplet":
        side = max(case["nx"], case["ny"])
        c = _droplet(rng, side, case["axi"], case.get("hysteresis", False), case.get("streaming", False))
        return [c.crop(case["nx"], case["ny"])]
    return [_droplet(rng, s, case["axi"], kind == "serve", case.get("streaming", False))
            for s in _sides(case)]


# -- one pass -----------------------------------------------------------------

def prepare(case, seed):
    problems = _problems(case, seed)
    precision = PRECISION[case["precision"]]
    state = {"case": case, "precision": precision}
    if case["kind"] == "serve":
        state["requests"] = [wl.Request(k, 0.0, p, case["steps"]) for k, p in enumerate(problems)]
        return state
    if case.get("slabs"):
        state["solver"] = eulbfs.Solver([], precision=precision)
        state["slots"] = state["solver"].add_split(problems[0], case["slabs"])
    else:
        state["solver"] = eulbfs.Solver(problems, precision=precision)
        state["slots"] = list(range(len(problems)))
    return state


def _which(case):
    # a conductive layer has no flow and no gas, layers along x no flow along y
    return {"stefan": ("H", "T", "Fl"), "layers": ("H", "T", "Fl", "C", "p", "u")}.get(
        case["kind"], ("H", "T", "Fl", "C", "p", "u", "v"))


def _reads_fields(case):
    return case["precision"] == "fp64" and case["kind"] != "batch"


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        report = serving.serve(state["requests"], precision=state["precision"], realtime=False)
        return [o.diag for o in report.outcomes]
    solver = state["solver"]
    solver.step(case["steps"])
    if _reads_fields(case):
        return [solver.fields(s, _which(case)) for s in state["slots"]]
    dtype = np.float64 if case["precision"] == "fp64" else np.float32
    return [np.frombuffer(solver.save(s)[0], dtype=dtype) for s in state["slots"]]


def work(case):
    n = _cells(case) * case["steps"]
    return {"bytes": float(n * BYTES[case["precision"]]), "flops": float(n * FLOPS)}


# -- the method in 64 bits ------------------------------------------------------

E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
WT = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
CS2 = 1.0 / 3.0
G = 2   # ghost layers


class _Exact:
    """Domains of one shape and the same kinds of boundaries, stacked along the first axis."""

    def __init__(self, problems, device):
        a = problems[0]
        self.nx, self.ny, self.axi, self.bc = a.nx, a.ny, bool(a.axisymmetric), a.bc
        self.dev = device
        self.zsv = bool(a.props.zero_solid_velocity)
        base = [c.dt_stream for c in problems]
        self.dth, self.dtf, self.dtg = (self._v([getattr(c, k) or b for c, b in zip(problems, base)])
                                        for k in ("dt_h", "dt_f", "dt_g"))
        P = [c.props for c in problems]
        self.ph = {q: [self._v([getattr(getattr(p, k), q) for p in P]) for k in "slg"]
                   for q in ("rho", "mu", "lam", "cp")}
        self.L, self.Ts, self.Tl = (self._v([getattr(p, k) for p in P]) for k in ("L", "Ts", "Tl"))
        sigma, xi = self._v([p.sigma for p in P]), self._v([p.xi for p in P])
        self.xi, self.beta, self.kappa = xi, 12.0 * sigma / xi, 1.5 * xi * sigma
        self.tau_g = self._v([p.tau_g for p in P])
        self.Qg = self._v([p.Mc for p in P]) / ((self.tau_g - 0.5) * self.dtg)
        self.Cref = 0.5 * (self.ph["cp"][0] + self.ph["cp"][1])
        self.kv = 1.0 - self.ph["rho"][0] / self.ph["rho"][1]
        self.gx, self.gy = self._v([p.gx for p in P]), self._v([p.gy for p in P])
        self.dt = self._v([c.dt for c in problems])
        side = lambda f: {k: self._v([f(getattr(c.bc, k)) for c in problems])  # noqa: E731
                          for k in ("xlo", "xhi", "ylo", "yhi")}
        cos = lambda deg: math.cos(deg * math.pi / 180.0)  # noqa: E731
        self.Tw = side(lambda s: s.Tw)
        self.ceq, self.cadv, self.crec = (side(lambda s: cos(s.theta_deg)), side(lambda s: cos(s.theta_adv_deg)),
                                          side(lambda s: cos(s.theta_rec_deg)))
        self.per_x, self.per_y = a.bc.xlo.thermal == wl.PERIODIC, a.bc.ylo.thermal == wl.PERIODIC
        F = {k: torch.stack([torch.from_numpy(np.asarray(c.init[k], dtype=np.float64)) for c in problems]).to(device)
             for k in ("T", "Fl", "C", "u", "v", "p")}
        C = F["C"]
        cps, cpl, Hs, Hl = self._branches(C.clamp(0, 1))
        f = torch.where(self.Tl > self.Ts, (F["T"] - self.Ts) / (self.Tl - self.Ts).clamp_min(1e-300), F["Fl"])
        H = torch.where(F["T"] < self.Ts, cps * F["T"],
                        torch.where(F["T"] > self.Tl, Hl + cpl * (F["T"] - self.Tl),
                                    Hs + f.clamp(0, 1) * (Hl - Hs)))
        rho = self._mixed(C, self._enthalpy(H, C)[1])["rho"]
        self.W = [H, F["p"], rho * CS2 * F["u"], rho * CS2 * F["v"], C]
        self.Fsp = 1.0 - self._enthalpy(H, C)[1]

    def _v(self, x):
        return torch.tensor(x, dtype=torch.float64, device=self.dev).reshape(-1, 1, 1)

    def _branches(self, Ct):
        s, l, g = self.ph["cp"]
        cps, cpl = Ct * s + (1 - Ct) * g, Ct * l + (1 - Ct) * g
        return cps, cpl, cps * self.Ts, cpl * self.Tl + self.L

    def _enthalpy(self, H, C):
        cps, cpl, Hs, Hl = self._branches(C.clamp(0, 1))
        f = (H - Hs) / (Hl - Hs)
        solid, liquid = H < Hs, H > Hl
        Fl = torch.where(solid, 0.0, torch.where(liquid, 1.0, f))
        T = torch.where(solid, H / cps, torch.where(liquid, self.Tl + (H - Hl) / cpl, self.Ts + f * (self.Tl - self.Ts)))
        return T, Fl

    def _mixed(self, C, Fl):
        Ct = C.clamp(0, 1)
        return {q: Ct * ((1 - Fl) * s + Fl * l) + (1 - Ct) * g for q, (s, l, g) in self.ph.items()}

    def _cos_theta(self, side, a, t):
        """The angle's cosine at the wall positions `t` of `side`: the fixed
        one, or the apparent one clamped to the hysteresis window; `a` is C
        without ghosts along the wall's normal, walls along y last."""
        if getattr(self.bc, side).phase != wl.WETTING_HYST:
            return self.ceq[side]
        lo = side in ("xlo", "ylo")
        c0, c1 = (a[..., 0], a[..., 1]) if lo else (a[..., -1], a[..., -2])
        n = c0.shape[-1]
        per = self.per_y if side[0] == "x" else self.per_x
        k = torch.arange(n, device=self.dev)
        kp, km = ((k + 1) % n, (k - 1) % n) if per else ((k + 1).clamp_max(n - 1), (k - 1).clamp_min(0))
        dt = (c0[..., kp] - c0[..., km]) / (2.0 if per else (kp - km))
        dn = c0 - c1
        g = torch.sqrt(dn * dn + dt * dt)
        apparent = torch.minimum(torch.maximum(dn / g.clamp_min(1e-300), self.cadv[side][..., 0]), self.crec[side][..., 0])
        wall = torch.where((c0 * (1 - c0) >= 1e-3) & (g > 0), apparent, self.ceq[side][..., 0])
        return wall[..., (t % n) if per else t.clamp(0, n - 1)]

    def _rule(self, side, name, k, v, cos):
        s = getattr(self.bc, side)
        normal = "u" if side[0] == "x" else "v"
        if name == "T" and s.thermal == wl.DIRICHLET_T:
            return 2.0 * self.Tw[side][..., 0] - v
        if name == "p" and s.flow == wl.OUTLET:
            return -v
        if name in "uv" and (s.flow == wl.NOSLIP or (s.flow == wl.SYMMETRY and name == normal)):
            return -v
        if name == "C" and s.phase in (wl.WETTING, wl.WETTING_HYST):
            c = cos if cos.dim() == 2 else cos[..., 0]
            return v + (2 * k - 1) * (4.0 * c / self.xi[..., 0]) * v * (1 - v)
        return v

    def _pad(self, name, a, C):
        """a with two ghost layers on every side: x sides first, then y."""
        B, ny, nx = a.shape
        out = a.new_empty(B, ny + 2 * G, nx + 2 * G)
        out[:, G:-G, G:-G] = a
        rows, cols = torch.arange(ny, device=self.dev), torch.arange(-G, nx + G, device=self.dev)
        cos = lambda side: self._cos_theta(side, C if side[0] == "x" else C.transpose(1, 2),  # noqa: E731
                                           rows if side[0] == "x" else cols) if name == "C" else None
        cx, cy = [cos("xlo"), cos("xhi")], [cos("ylo"), cos("yhi")]
        for k in range(1, G + 1):
            if self.per_x:
                lo, hi = a[:, :, nx - k], a[:, :, k - 1]
            else:
                lo, hi = self._rule("xlo", name, k, a[:, :, k - 1], cx[0]), self._rule("xhi", name, k, a[:, :, nx - k], cx[1])
            out[:, G:-G, G - k], out[:, G:-G, G + nx - 1 + k] = lo, hi
        for k in range(1, G + 1):
            # a periodic axis of fewer rows than ghost layers wraps more than once
            near, far = out[:, G + (k - 1) % ny], out[:, G + (ny - k) % ny]
            if self.per_y:
                lo, hi = far, near
            else:
                lo, hi = self._rule("ylo", name, k, near, cy[0]), self._rule("yhi", name, k, far, cy[1])
            out[:, G - k], out[:, G + ny - 1 + k] = lo, hi
        return out

    def _faces(self, P, rf):
        """Flux moments of the faces across the last axis; P: padded fields
        with "n" and "t" the normal and tangential velocity, rf: radii of the
        faces for the axisymmetric mass source on the radial velocity `r`."""
        F = {f: a for f, a in P.items() if f not in "ruv"}
        val = {f: a[:, G:-G, 1:-1] for f, a in F.items()}
        gn = {f: 0.5 * (a[:, G:-G, 2:] - a[:, G:-G, :-2]) for f, a in F.items()}
        gt = {f: 0.5 * (a[:, G + 1:-G + 1, 1:-1] - a[:, G - 1:-G - 1, 1:-1]) for f, a in F.items()}

        def at(f, en, et, d):
            lo, hi = (..., slice(None, -1)), (..., slice(1, None))
            left = lambda off: val[f][lo] + off * gn[f][lo] - et * d * gt[f][lo]  # noqa: E731
            right = lambda off: val[f][hi] - off * gn[f][hi] - et * d * gt[f][hi]  # noqa: E731
            if en > 0:
                return left(0.5 - d)
            if en < 0:
                return right(0.5 - d)
            return 0.5 * (left(0.5) + right(0.5))

        face = {f: at(f, 0, 0, 0.0) for f in ("rho", "T", "cp", "lam", "mu", "muc")}
        rho_f = face["rho"]
        src = 0.0
        if rf is not None:
            inv = torch.where(rf > 0, 1.0 / rf.clamp_min(0.5), 0.0)
            src = -self.dtf * rho_f * CS2 * at(P["r"], 0, 0, 0.0) * inv
        p_f = mn = mt = C_f = 0.0
        h_n = fm_nn = fm_nt = g_n = 0.0
        for (en, et), w in zip(E, WT):
            un, ut = at("n", en, et, self.dth), at("t", en, et, self.dth)
            eu = en * un + et * ut
            q = eu / CS2 + eu * eu / (2 * CS2 * CS2) - (un * un + ut * ut) / (2 * CS2)
            if en:
                cp, T = at("cp", en, et, self.dth), at("T", en, et, self.dth)
                h_n = h_n + en * w * cp * T * (self.Cref / cp + q)
            if self.same:
                un_f, ut_f, eu_f, q_f, eu_g = un, ut, eu, q, eu
            else:
                un_f, ut_f = at("n", en, et, self.dtf), at("t", en, et, self.dtf)
                eu_f = en * un_f + et * ut_f
                q_f = eu_f / CS2 + eu_f * eu_f / (2 * CS2 * CS2) - (un_f * un_f + ut_f * ut_f) / (2 * CS2)
                eu_g = en * at("n", en, et, self.dtg) + et * at("t", en, et, self.dtg)
            p, rho = at("p", en, et, self.dtf), at("rho", en, et, self.dtf)
            feq = w * (p + rho * CS2 * q_f) + w * src
            p_f = p_f + feq
            if en:
                fm = w * (p + rho_f * CS2 * q_f) + w * src
                mn, fm_nn, fm_nt = mn + en * feq, fm_nn + fm, fm_nt + en * et * fm
            if et:
                mt = mt + et * feq
            C, muc = at("C", en, et, self.dtg), at("muc", en, et, self.dtg)
            geq = w * (muc * self.Qg + C * eu_g) / CS2 if (en or et) else C - muc * self.Qg * (1 - w) / CS2
            C_f = C_f + geq
            if en:
                g_n = g_n + en * geq
        un, ut = mn / (rho_f * CS2), mt / (rho_f * CS2)
        th = face["lam"] / (rho_f * self.Cref * CS2 * self.dth)   # tau - 1/2 of h, f, g
        tf = face["mu"] / (rho_f * CS2 * self.dtf)
        tg = self.tau_g - 0.5
        return ((1 - th) * face["cp"] * face["T"] * un + th * h_n, rho_f * CS2 * un,
                (1 - tf) * CS2 * (p_f + rho_f * un * un) + tf * fm_nn,
                (1 - tf) * CS2 * rho_f * un * ut + tf * fm_nt,
                (1 - tg) * C_f * un + tg * g_n, un)

    def _residual(self, W, dFs):
        H, p, mx, my, C = W
        T, Fl = self._enthalpy(H, C)
        prim = self._mixed(C, Fl)
        rho = prim["rho"]
        prim.update(T=T, p=p, u=mx / (rho * CS2), v=my / (rho * CS2), C=C)
        P = {f: self._pad(f, a, C) for f, a in prim.items()}
        c = P["C"]
        mid = c[:, G:-G, G:-G]
        e, w, n, s = c[:, G:-G, G + 1:-G + 1], c[:, G:-G, G - 1:-G - 1], c[:, G + 1:-G + 1, G:-G], c[:, G - 1:-G - 1, G:-G]
        rw = torch.arange(self.nx, dtype=torch.float64, device=self.dev)
        rc, re = rw + 0.5, rw + 1.0
        lap = ((re * (e - mid) - rw * (mid - w)) / rc if self.axi else e + w - 2 * mid) + n + s - 2 * mid
        muc = 2 * self.beta * C * (C - 1) * (2 * C - 1) - self.kappa * lap
        P["muc"] = self._pad("muc", muc, C)
        rf = torch.arange(self.nx + 1, dtype=torch.float64, device=self.dev)
        fx = self._faces(dict(P, n=P["u"], t=P["v"], r="n"), rf if self.axi else None)
        Pt = {f: a.transpose(1, 2) for f, a in P.items()}
        fy = self._faces(dict(Pt, n=Pt["v"], t=Pt["u"], r="t"), rc[:, None] if self.axi else None)
        fy = [f.transpose(1, 2) for f in fy]
        fx, fy = list(fx), [fy[0], fy[1], fy[3], fy[2], fy[4], fy[5]]   # both as (h, p, mx, my, C, u_n)
        div = []
        for a, b in zip(fx, fy):
            dx = (rf[1:] * a[..., 1:] - rf[:-1] * a[..., :-1]) / rc if self.axi else a[..., 1:] - a[..., :-1]
            div.append(dx + b[:, 1:] - b[:, :-1])
        gx = lambda f: 0.5 * (P[f][:, G:-G, G + 1:-G + 1] - P[f][:, G:-G, G - 1:-G - 1])  # noqa: E731
        gy = lambda f: 0.5 * (P[f][:, G + 1:-G + 1, G:-G] - P[f][:, G - 1:-G - 1, G:-G])  # noqa: E731
        u, v, D = prim["u"], prim["v"], C.clamp(0, 1) * dFs
        R = [-div[0] + prim["cp"] * T * div[5],
             -div[1] + CS2 * (u * gx("rho") + v * gy("rho")) + rho * CS2 * self.kv * D,
             -div[2] + CS2 * (-Fl * C * gx("muc") + rho * self.gx - rho * u * D),
             -div[3] + CS2 * (-Fl * C * gy("muc") + rho * self.gy - rho * v * D),
             -div[4] + C * self.kv * dFs]
        if self.axi:
            R[2] = R[2] + CS2 * (p - self.dtf * div[1] - 2 * prim["mu"] * u / rc) / rc
        return R

    def step(self):
        self.same = bool((self.dth == self.dtf).all() and (self.dth == self.dtg).all())
        Fs = 1.0 - self._enthalpy(self.W[0], self.W[4])[1]
        dFs = (Fs - self.Fsp) / self.dt
        Wn, cur = self.W, self.W
        for A, B, c in ((1.0, 0.0, 1.0), (0.75, 0.25, 0.25), (1 / 3, 2 / 3, 2 / 3)):
            R = self._residual(cur, dFs)
            cur = [A * a + B * b + c * self.dt * r for a, b, r in zip(Wn, cur, R)]
            if self.zsv:
                keep = 1.0 - cur[4].clamp(0, 1) * (1.0 - self._enthalpy(cur[0], cur[4])[1])
                cur[2], cur[3] = cur[2] * keep, cur[3] * keep
        self.W, self.Fsp = cur, Fs

    def fields(self, b):
        H, p, mx, my, C = (a[b:b + 1] for a in self.W)
        sub = lambda d: {k: [x[b:b + 1] for x in v] for k, v in d.items()}  # noqa: E731
        one = object.__new__(_Exact)
        one.ph, one.L, one.Ts, one.Tl = sub(self.ph), self.L[b:b + 1], self.Ts[b:b + 1], self.Tl[b:b + 1]
        T, Fl = one._enthalpy(H, C)
        m = one._mixed(C, Fl)["rho"] * CS2
        return {k: a[0] for k, a in dict(H=H, T=T, Fl=Fl, C=C, p=p, u=mx / m, v=my / m).items()}

    def planes(self, b, fp32c):
        """Checkpoint planes of domain b: the state in working precision, then F_s."""
        H, p, mx, my, C = (a[b] for a in self.W)
        if not fp32c:
            return [H, p, mx, my, C, self.Fsp[b]]
        pair = lambda x: [x.float().double(), x - x.float().double()]  # noqa: E731
        return pair(H) + [p, mx, my] + pair(C) + [self.Fsp[b]]

    def diag(self, b, steps, dt):
        f = self.fields(b)
        rho = ((f["C"].clamp(0, 1) * ((1 - f["Fl"]) * self.ph["rho"][0][b] + f["Fl"] * self.ph["rho"][1][b]))
               + (1 - f["C"].clamp(0, 1)) * self.ph["rho"][2][b])
        vol = (torch.arange(self.nx, dtype=torch.float64, device=self.dev) + 0.5) if self.axi else 1.0
        total = lambda x: float((vol * x).sum())  # noqa: E731
        phase, solid = total(f["C"]), total(f["C"].clamp(0, 1) * (1 - f["Fl"]))
        base = 0.5 * self.nx * self.nx if self.axi else self.ny
        return {"step": None, "t": steps * dt, "mass": total(rho), "enthalpy": total(f["H"]), "phase_vol": phase,
                "solid_vol": solid, "front_pos": solid / base, "interface_pos": phase / base,
                "max_speed": float(torch.sqrt(f["u"] ** 2 + f["v"] ** 2).max()), "nonfinite": None}


def exact(case, seed):
    if _cells(case) * case["steps"] > 2.0e8:
        return None   # minutes of plain torch operations
    problems = _problems(case, seed)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    fp32c = case["precision"] == "fp32c"
    shapes = {}
    for k, c in enumerate(problems):
        shapes.setdefault((c.ny, c.nx), []).append(k)
    out = [None] * len(problems)
    for ks in shapes.values():
        e = _Exact([problems[k] for k in ks], device)
        for _ in range(case["steps"]):
            e.step()
        for b, k in enumerate(ks):
            if case["kind"] == "serve":
                out[k] = e.diag(b, case["steps"], problems[k].dt)
            elif _reads_fields(case):
                f = e.fields(b)
                out[k] = {q: f[q].cpu() for q in _which(case)}
            else:
                out[k] = [a.cpu() for a in e.planes(b, fp32c)]
    if case["kind"] == "serve" or _reads_fields(case):
        return out
    if not case.get("slabs"):
        return [torch.stack(p).reshape(-1) for p in out]
    # a slab's planes hold three rows of each neighbour; its F_s only its own
    n, ny = case["slabs"], case["ny"]
    slabs = []
    for i in range(n):
        y0, y1 = i * ny // n, (i + 1) * ny // n
        lo, hi = 3 if i else 0, 3 if i < n - 1 else 0
        rows = [a[y0 - lo:y1 + hi] for a in out[0]]
        rows[-1] = torch.zeros_like(rows[-1])
        rows[-1][lo:lo + y1 - y0] = out[0][-1][y0:y1]
        slabs.append(torch.stack(rows).reshape(-1))
    return slabs
