"""What is measured of this framework, over the ranges that its users run it in.

The framework advances atmospheric columns of a stiff photochemical network: controlled implicit steps
in FP64 and in mixed precision, one column at a time or many in a batch; and around them the radiation
field, the chemical-equilibrium start, the pathway analyser and the Lagrangian parcel sweep.  The cases
call these through the public Column and Batch classes on seeded synthetic networks of the sizes that
the benchmark and the tests use (20 to 594 species, 40 to 200 layers, 1,000 and 10,000 wavelength bins).

exact() states the same results in plain torch, FP64, without the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2512_06729_gb300 import synth, xk

# two-body, three-body, photolysis reactions and element set of the networks in use
_NETWORKS = {20: (60, 0, 0, "cho"), 96: (960, 240, 40, "chons"), 250: (2600, 650, 80, "full"),
             594: (6016, 1504, 200, "full")}


def listed():
    return [
        # the smallest column there is (the textbook size), plain FP64: latency of a step
        dict(name="steps_tiny_fp64", kind="steps", species=20, layers=40, precision="fp64", start="user",
             dt0=1e-8, steps=8),
        # a C-H-O-N-S column in plain FP64: the accurate path at an ordinary size
        dict(name="steps_chons_fp64", kind="steps", species=96, layers=150, precision="fp64", start="user",
             dt0=1e-8, steps=4),
        # the same column in mixed precision: the ordinary run
        dict(name="steps_chons_mixed", kind="steps", species=96, layers=150, precision="mixed", start="user",
             dt0=1e-8, steps=8),
        # a sweep column of odd height, continued from chemical equilibrium at a later step size
        dict(name="steps_sweep_mixed", kind="steps", species=250, layers=137, precision="mixed",
             start="equilibrium", dt0=1e-4, steps=4),
        # the largest network, mixed: the headline step
        dict(name="steps_full_mixed", kind="steps", species=594, layers=150, precision="mixed", start="user",
             dt0=1e-8, steps=4),
        # the largest network in plain FP64: one linear step
        dict(name="delta_full_fp64", kind="delta", species=594, layers=150, precision="fp64", start="user", dt=1e-2),
        # serving: uneven columns advanced together, one round after another
        dict(name="batch_uneven_mixed", kind="batch", small=5, middle=2, large=1, rounds=2),
        # photolysis rates of the direct beam on the benchmark's grid, once per step of every run
        dict(name="photolysis_direct", kind="photolysis", species=594, layers=150, bins=1000, diffuse=0),
        # photolysis rates with scattering and the diffuse field on the fine grid
        dict(name="photolysis_diffuse", kind="photolysis", species=594, layers=150, bins=10000, diffuse=1),
        # the equilibrium composition every served request may start from
        dict(name="equilibrium_full", kind="equilibrium", species=594, layers=150),
        # reaction fluxes and fastest routes from eight species, the analysis of a finished run
        dict(name="pathways_full", kind="pathways", species=594, layers=150, sources=8),
        # one global iteration of the parcel scheme on a test-sized column
        dict(name="parcel_small", kind="parcel", species=40, layers=60),
    ]


def draw(rng):
    species = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["steps", "steps", "steps", "delta", "batch", "photolysis", "equilibrium", "pathways", "parcel"])
    layers = rng.randint(40, 150)
    if kind == "steps":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        start = rng.choice(["user", "equilibrium"])
        return dict(kind=kind, species=species(24, 594 if precision == "mixed" else 130), layers=layers,
                    precision=precision, start=start,
                    dt0=10.0 ** rng.uniform(-8, -6 if start == "user" else -3), steps=rng.randint(1, 4))
    if kind == "delta":
        precision = rng.choice(["mixed", "fp64"])
        return dict(kind=kind, species=species(24, 594 if precision == "mixed" else 300), layers=layers,
                    precision=precision, start="user", dt=10.0 ** rng.uniform(-8, -2))
    if kind == "batch":
        return dict(kind=kind, small=rng.randint(2, 6), middle=rng.randint(0, 2), large=rng.randint(0, 1),
                    rounds=rng.randint(1, 2))
    if kind == "photolysis":
        return dict(kind=kind, species=species(40, 594), layers=layers, bins=species(300, 10000),
                    diffuse=rng.randint(0, 1))
    if kind == "equilibrium":
        return dict(kind=kind, species=species(24, 594), layers=layers)
    if kind == "pathways":
        return dict(kind=kind, species=species(40, 594), layers=layers, sources=rng.randint(1, 8))
    return dict(kind=kind, species=species(24, 64), layers=rng.randint(20, 60))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _counts(S):
    if S in _NETWORKS:
        return _NETWORKS[S]
    if S < 90:
        return 3 * S, 3 * S // 4, max(S // 4, 1), "chons"
    return 8 * S, 2 * S, S // 3, "full" if S > 110 else "chons"


@functools.lru_cache(maxsize=16)
def _network(S, bins=1000, diffuse=0):
    """A network of S species on the standard profile (a data file of a user's program)."""
    n_two, n_three, n_photo, elements = _counts(S)
    for seed in range(40):
        try:
            prob = synth.make_problem(f"column-{S}sp", S, n_two, n_three, n_photo, synth.CONFIG_ELEMENTS[elements],
                                      synth.profile_tiny(40) if S == 20 else synth.profile_hot_jupiter(150), seed,
                                      W=1000 if diffuse else bins)
            break
        except RuntimeError:
            continue
    if diffuse:
        prob = synth.with_scattering(prob, albedo=0.1, diffuse=1, bins=bins)
    return prob


def _problem(S, L, seed, bins=1000, diffuse=0):
    """That network in an atmosphere of L layers, its temperature, mixing and composition from the seed."""
    rng = np.random.default_rng([seed, S, L])
    net = _network(S, bins, diffuse)
    if S == 20:
        P, T, Kzz = synth.profile_tiny(L)
        T = T * rng.uniform(0.97, 1.03)
    else:
        P, T, Kzz = synth.profile_hot_jupiter(L, T_scale=rng.uniform(0.9, 1.1), Kzz_scale=10.0 ** rng.uniform(-0.3, 0.3))
    f = 10.0 ** rng.uniform(-10.0, -5.0, size=S)
    f[0] = 0.85
    f[1] = 0.0
    f[1] = max(0.15 - f[2:].sum(), 1e-3)
    # abundances that vary with height, as in an atmosphere that has evolved
    f = np.tile(f, (L, 1)) * (1.0 + 0.2 * rng.uniform(-1.0, 1.0, size=(L, 1)) * (np.arange(S) > 1))
    return net.replace(P_bar=P, T=T, Kzz=Kzz, f0=f)


def _column(case, seed):
    prob = _problem(case["species"], case["layers"], seed, case.get("bins", 1000), case.get("diffuse", 0))
    return prob, xk.Column(prob, precision=case.get("precision", "fp64"))


def _start(col, prob, start):
    """The start state: the given composition, or chemical equilibrium at its element totals."""
    col.set_mixing_ratios(prob.f0)
    if start == "equilibrium":
        col.equilibrium(set_state=True)
    return col.get_state(device=True)


_BATCH_SPECIES = {"small": 96, "middle": 250, "large": 594}


def _batch_columns(case):
    """(species, layers) of the batch's columns: layers uneven between 80 and 200."""
    out = []
    for what, S in _BATCH_SPECIES.items():
        for i in range(case[what]):
            out.append((S, 80 + (37 * i + S) % 121))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cols, starts = [], []
        batch = xk.Batch(200 * 2 ** 30, len(_batch_columns(case)))
        for i, (S, L) in enumerate(_batch_columns(case)):
            prob = _problem(S, L, 1000 * seed + i)
            col = xk.Column(prob, precision="mixed")
            starts.append(_start(col, prob, "user"))
            batch.add(col, dt0=1e-8)
            cols.append(col)
        return dict(case=case, batch=batch, cols=cols, starts=starts)
    prob, col = _column(case, seed)
    state = dict(case=case, col=col, n=_start(col, prob, case.get("start", "user")))
    if kind == "pathways":
        rng = np.random.default_rng([seed, 7])
        state["sources"] = 2 + rng.choice(case["species"] - 2, size=case["sources"], replace=False)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        for col, n in zip(state["cols"], state["starts"]):
            col.set_state(n)
        for _ in range(case["rounds"]):
            state["batch"].step(1)
        return [col.get_state(device=True) for col in state["cols"]]
    col, n = state["col"], state["n"]
    if kind == "steps":
        col.set_state(n)
        col.run_to_steady(dt0=case["dt0"], max_steps=case["steps"])
        return col.get_state(device=True)
    if kind == "delta":
        return col.step_delta(n, case["dt"])[0]
    if kind == "photolysis":
        return col.eval_photolysis(n)
    if kind == "equilibrium":
        return col.equilibrium()[0]
    if kind == "pathways":
        q = col.reaction_fluxes(n)
        return dict(col.pathways(q, state["sources"]), q=q)
    col.set_state(n)
    col.parcel_iteration(h=1e-8)
    return col.get_state(device=True)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        total = dict(bytes=0.0, flops=0.0)
        for S, L in _batch_columns(case):
            w = work(dict(kind="steps", species=S, layers=L, steps=case["rounds"]))
            total = {k: total[k] + w[k] for k in total}
        return total
    S, L, kind = case["species"], case["layers"], case["kind"]
    n_two, n_three, n_photo, _ = _counts(S)
    R, W = n_two + n_three + n_photo, case.get("bins", 1000) if n_photo else 0
    absorbers = min(S, n_photo)
    scatterers = S // 3 if case.get("diffuse") else 0
    photo_bytes = 8.0 * ((absorbers + scatterers + n_photo) * W + L * n_photo)
    photo_flops = 2.0 * L * W * (absorbers + scatterers + n_photo)
    if kind in ("steps", "delta"):
        # rate coefficients and the state in, the state out; photolysis, the rates with their
        # derivatives, and the block elimination (each layer's Schur complement takes the whole
        # inverse of its neighbour's block)
        steps = case.get("steps", 1)
        return dict(bytes=8.0 * (2 * L * S + 2 * L * R) + photo_bytes,
                    flops=steps * (L * 2.0 * S ** 3 + photo_flops + 40.0 * L * R))
    if kind == "photolysis":
        return dict(bytes=8.0 * L * S + photo_bytes, flops=photo_flops)
    if kind == "equilibrium":
        # about 20 Newton iterations over the species that hold each element pair
        return dict(bytes=8.0 * 2 * L * S, flops=20.0 * L * S * 60)
    if kind == "pathways":
        nsrc = case["sources"]
        return dict(bytes=8.0 * (L * S + 4 * L * R) + photo_bytes + nsrc * L * S * 28.0,
                    flops=photo_flops + 6.0 * L * R + nsrc * L * 7.0 * R * 2)
    # parcel: the visits' implicit steps, about eight to a visit
    return dict(bytes=8.0 * (2 * L * S + 2 * L * R), flops=(2 * L - 1) * 8 * (2.0 / 3.0 * S ** 3 + 6.0 * S * S + 40.0 * R))


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
_KB, _AMU = 1.380649e-16, 1.66053906660e-24


class _Exact:
    """The column's equations written out: rates, photolysis, residual, Jacobian, implicit step."""

    def __init__(self, p):
        self.p = p
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=self.dev)
        self.t = t
        S, L, R = p.S, p.L, p.R
        self.S, self.L, self.R = S, L, R
        T = p.T
        self.ngas = p.P_bar * 1e6 / (_KB * T)
        # hydrostatic grid
        Th = 0.5 * (T[:-1] + T[1:])
        H = _KB * Th / (p.mbar * _AMU * p.g)
        self.z = np.concatenate([[0.0], np.cumsum(H * np.log(p.P_bar[:-1] / p.P_bar[1:]))])
        h = np.diff(self.z)
        dz = np.empty(L)
        dz[0], dz[-1] = h[0], h[-1]
        dz[1:-1] = 0.5 * (self.z[2:] - self.z[:-2])
        self.dz = t(dz)[:, None]
        # interface coefficients
        nh = 0.5 * (self.ngas[:-1] + self.ngas[1:])
        Kh = 0.5 * (p.Kzz[:-1] + p.Kzz[1:])
        D = p.dcoef[None, :] * (Th ** 0.75 / nh)[:, None]
        Hy = (_KB * Th)[:, None] / (p.mass[None, :] * _AMU * p.g)
        a = 1.0 / Hy + ((1.0 + p.alpha_T) * np.diff(T) / h / Th)[:, None]
        self.u = t((Kh * nh / (h * self.ngas[:-1]))[:, None] + D * (1.0 / h[:, None] - 0.5 * a))
        self.v = t((Kh * nh / (h * self.ngas[1:]))[:, None] + D * (1.0 / h[:, None] + 0.5 * a))
        self.ng = t(self.ngas)[:, None]
        # Gibbs energies, rate coefficients
        a7 = np.where((T[:, None] < p.nasa[None, :, 0])[:, :, None], p.nasa[None, :, 1:8], p.nasa[None, :, 8:15])
        TT = T[:, None]
        self.grt = (a7[..., 0] * (1.0 - np.log(TT)) - a7[..., 1] * TT / 2 - a7[..., 2] * TT ** 2 / 6
                    - a7[..., 3] * TT ** 3 / 12 - a7[..., 4] * TT ** 4 / 20 + a7[..., 5] / TT - a7[..., 6])
        self.reac, self.prod = p.reac, p.prod
        pad = np.concatenate([self.grt, np.zeros((L, 1))], axis=1)
        dG = pad[:, p.prod].sum(axis=2) - pad[:, p.reac].sum(axis=2)
        dnu = (p.prod >= 0).sum(axis=1) - (p.reac >= 0).sum(axis=1)
        lnk = -dG + dnu[None, :] * np.log(1e6 / (_KB * TT))
        Tb = np.where(p.form[None, :] == 0, TT / 300.0, TT)
        arr = lambda i: p.arr[None, :, i] * Tb ** p.arr[None, :, i + 1] * np.exp(-p.arr[None, :, i + 2] / TT)
        two, three = p.rtype == 0, p.rtype == 1
        kf = np.zeros((L, R))
        kf[:, two] = arr(0)[:, two]
        if three.any():
            k0, ki = arr(3)[:, three], arr(6)[:, three]
            M = self.ngas[:, None]
            Pr = k0 * M / ki
            tr = p.troe[three][None]
            safe = np.where(tr == 0.0, 1.0, tr)
            Fc = (1 - tr[..., 0]) * np.exp(-TT / safe[..., 1]) + tr[..., 0] * np.exp(-TT / safe[..., 2])
            Fc = Fc + np.where(tr[..., 3] != 0.0, np.exp(-tr[..., 3] / TT), 0.0)
            broad = (tr[..., 0] != 0.0) & (Pr > 0.0)
            lF = np.log10(np.where(broad, Fc, 1.0))
            x = np.log10(np.where(broad, Pr, 1.0)) + (-0.4 - 0.67 * lF)
            q = x / (0.75 - 1.27 * lF - 0.14 * x)
            kf[:, three] = k0 * M / (1 + Pr) * np.where(broad, 10.0 ** (lF / (1 + q * q)), 1.0)
        kr = np.where((p.rtype == 2)[None, :], 0.0, kf / np.exp(lnk))
        self.kf, self.kr = t(kf), t(kr)
        self.photo = torch.as_tensor(np.flatnonzero(p.rtype == 2), device=self.dev)
        # index lists: (row, column, reaction, slot, sign) of the Jacobian, and the stoichiometry
        slots = np.concatenate([p.reac, p.prod], axis=1)
        self.slots = torch.as_tensor(np.where(slots < 0, S, slots), device=self.dev).long()
        rr, qq = np.nonzero(slots >= 0)
        self.st = [torch.as_tensor(x, device=self.dev).long() for x in (slots[rr, qq], rr)]
        self.st_sign = t(np.where(qq < 3, -1.0, 1.0))

    def photolysis(self, n):
        p = self.p
        if p.Rph == 0:
            return torch.zeros((self.L, 0), dtype=torch.float64, device=self.dev)
        ta = (n @ self.t(p.sigma_abs)) * self.dz
        ts = (n @ self.t(p.sigma_s)) * self.dz if p.sigma_s is not None else torch.zeros_like(ta)
        dt = ta + ts
        top = torch.flip(torch.cumsum(torch.flip(dt, [0]), 0), [0]) - dt      # optical depth above each layer
        J0 = self.t(p.J0)[None, :]
        J = J0 * torch.exp(-(top + 0.5 * dt) / p.mu)
        if p.diffuse:
            om = torch.where(dt > 0, ts / torch.where(dt > 0, dt, torch.ones_like(dt)), torch.zeros_like(dt))
            t = torch.exp(-2.0 * dt)
            r = (1 - t) * om / 2
            Tr = t + r
            src = 0.5 * om * p.mu * J0 * (torch.exp(-top / p.mu) - torch.exp(-(top + dt) / p.mu))
            L = self.L
            refl = torch.zeros((L + 1, J.shape[1]), dtype=torch.float64, device=self.dev)   # layers from k up
            emit = torch.zeros_like(refl)
            for k in range(L - 1, -1, -1):
                den = 1 - r[k] * refl[k + 1]
                refl[k] = r[k] + Tr[k] * refl[k + 1] * Tr[k] / den
                emit[k] = Tr[k] * (emit[k + 1] + refl[k + 1] * (r[k] * emit[k + 1] + src[k]) / den) + src[k]
            beam = p.mu * J0[0] * torch.exp(-(top[0] + dt[0]) / p.mu)
            U = p.albedo * (emit[0] + beam) / (1 - p.albedo * refl[0])
            for k in range(L):
                Dk = refl[k] * U + emit[k]
                Un = (Tr[k] * U + r[k] * emit[k + 1] + src[k]) / (1 - r[k] * refl[k + 1])
                Dn = refl[k + 1] * Un + emit[k + 1]
                J[k] += 0.25 * (U + Un + Dk + Dn)
                U = Un
        return p.tf * (J * self.t(p.dlam)[None, :]) @ self.t(p.sigma).T

    def terms(self, n):
        """Forward and reverse rates [L, R] and the six partial derivatives [L, R, 6]."""
        kf = self.kf.clone()
        if len(self.photo):
            kf[:, self.photo] = self.photolysis(n)[:, torch.as_tensor(self.p.prow, device=self.dev)[self.photo].long()]
        one = torch.ones((self.L, 1), dtype=torch.float64, device=self.dev)
        x = torch.cat([n, one], 1)[:, self.slots]
        f, b = x[..., :3], x[..., 3:]
        wf, wb = kf * f.prod(-1), self.kr * b.prod(-1)
        d = torch.empty_like(x)
        for s in range(3):
            o = [q for q in range(3) if q != s]
            d[..., s] = kf * f[..., o[0]] * f[..., o[1]]
            d[..., 3 + s] = -self.kr * b[..., o[0]] * b[..., o[1]]
        return wf, wb, d

    def residual(self, n, w):
        F = torch.zeros_like(n).index_add_(1, self.st[0], self.st_sign * w[:, self.st[1]])
        phi = self.u * n[:-1] - self.v * n[1:]
        F[:-1] -= phi / self.dz[:-1]
        F[1:] += phi / self.dz[1:]
        return F

    def delta(self, n, dt):
        """The solution of (I/dt - J(n)) delta = F(n): block elimination and three refinement sweeps."""
        S, L = self.S, self.L
        wf, wb, d = self.terms(n)
        F = self.residual(n, wf - wb)
        s = torch.maximum(n, 1e-20 * self.ng)
        A = torch.zeros((L, S * (S + 1)), dtype=torch.float64, device=self.dev)
        for q in range(6):
            cols = self.slots[self.st[1], q]
            A.index_add_(1, self.st[0] * (S + 1) + cols, -self.st_sign * d[:, self.st[1], q])
        A = A.view(L, S, S + 1)[..., :S]
        dg = torch.full_like(n, 1.0 / dt)
        dg[:-1] += self.u / self.dz[:-1]
        dg[1:] += self.v / self.dz[1:]
        A = A * s[:, None, :] / s[:, :, None] + torch.diag_embed(dg)
        lo, up = torch.zeros_like(n), torch.zeros_like(n)
        lo[1:] = -self.u / self.dz[1:] * s[:-1] / s[1:]
        up[:-1] = -self.v / self.dz[:-1] * s[1:] / s[:-1]
        eye = torch.eye(S, dtype=torch.float64, device=self.dev)
        lus, inv = [], None
        for k in range(L):
            B = A[k] if inv is None else A[k] - lo[k][:, None] * inv * up[k - 1][None, :]
            lu = torch.linalg.lu_factor(B)
            lus.append(lu)
            inv = torch.linalg.lu_solve(*lu, eye)

        def solve(r):
            g, x = torch.empty_like(r), torch.empty_like(r)
            for k in range(L):
                rk = r[k] if k == 0 else r[k] - lo[k] * g[k - 1]
                g[k] = torch.linalg.lu_solve(*lus[k], rk[:, None])[:, 0]
            x[L - 1] = g[L - 1]
            for k in range(L - 2, -1, -1):
                x[k] = g[k] - torch.linalg.lu_solve(*lus[k], (up[k] * x[k + 1])[:, None])[:, 0]
            return x

        b = F / s
        x = solve(b)
        for _ in range(3):
            y = torch.bmm(A, x[:, :, None])[:, :, 0]
            y[1:] += lo[1:] * x[:-1]
            y[:-1] += up[:-1] * x[1:]
            x = x + solve(b - y)
        return x * s

    def steps(self, n, dt, count):
        """Controlled steps: reject on negative densities or a relative change above 1."""
        for _ in range(count):
            dl = self.delta(n, dt)
            nn = n + dl
            big = n > 1e-20 * self.ng
            rel = float((dl.abs() / n)[big].max())
            if bool((nn < -1e-12 * self.ng).any()) or not math.isfinite(rel) or rel > 1.0:
                dt *= 0.5
                continue
            n = nn.clamp_min(0.0)
            dt = min(dt * min(max(0.5 / rel if rel > 0 else 3.0, 0.5), 3.0), 1e8)
        return n

    def equilibrium(self, n):
        """Mole fractions of the Gibbs minimum at the element totals of n (Newton on the potentials)."""
        p = self.p
        E = p.E
        a = self.t(p.elem)
        b = n @ a
        b = b / b.sum(1, keepdim=True)
        g = self.t(self.grt) + self.t(np.log(p.P_bar))[:, None]
        lnN = torch.full_like(g, -math.log(p.S))
        lt = torch.zeros((self.L, 1), dtype=torch.float64, device=self.dev)
        pi = None
        for _ in range(400):
            N, tot = torch.exp(lnN), torch.exp(lt)
            mu = g + lnN - lt
            M = torch.zeros((self.L, E + 1, E + 1), dtype=torch.float64, device=self.dev)
            M[:, :E, :E] = torch.einsum("ky,ye,yf->kef", N, a, a)
            c = N @ a
            M[:, :E, E] = c
            M[:, E, :E] = c
            M[:, E, E] = N.sum(1) - tot[:, 0]
            rhs = torch.cat([b - c + (N * mu) @ a, (tot[:, 0] - N.sum(1) + (N * mu).sum(1))[:, None]], 1)
            sol = torch.linalg.solve(M, rhs[:, :, None])[:, :, 0]
            pi, dt = sol[:, :E], sol[:, E:]
            d = -mu + dt + pi @ a.T
            lx = lnN - lt
            major = lx > math.log(1e-8)
            big = torch.maximum(5 * dt.abs(), (d.abs() * major).max(1, keepdim=True).values)
            lam = torch.where(big > 2.0, 2.0 / big, torch.ones_like(big))
            grow = (~major) & (d - dt > 0)
            cap = torch.where(grow, ((-lx - 9.2103) / torch.where(grow, d - dt, torch.ones_like(d))).abs(), torch.ones_like(d))
            lam = torch.minimum(lam, cap.min(1, keepdim=True).values)
            lnN = lnN + lam * d
            lt = lt + lam * dt
            if float(((N * d.abs()).sum(1) / N.sum(1)).max()) < 1e-13 and float(dt.abs().max()) < 1e-13:
                break
        return torch.softmax(-g + pi @ a.T, 1)

    def distances(self, q, sources):
        """Least summed inverse rates from each source in every layer [nsrc, L, S] (relaxed to the end)."""
        S, L = self.S, self.L
        reac, prod = self.p.reac, self.p.prod
        fr, to, re, di = [], [], [], []
        for i in range(3):
            for j in range(3):
                ok = np.flatnonzero((reac[:, i] >= 0) & (prod[:, j] >= 0) & (reac[:, i] != prod[:, j]))
                fr += [reac[ok, i], prod[ok, j]]
                to += [prod[ok, j], reac[ok, i]]
                re += [ok, ok]
                di += [np.zeros_like(ok), np.ones_like(ok)]
        idx = lambda x: torch.as_tensor(np.concatenate(x).astype(np.int64), device=self.dev)
        fr, to, re, di = idx(fr), idx(to), idx(re), idx(di)
        inf = float("inf")
        w = torch.where(q > 0, 1.0 / q, torch.full_like(q, inf))[:, re, di]
        W = torch.full((L, S * S), inf, dtype=torch.float64, device=self.dev)
        W = W.scatter_reduce(1, (fr * S + to).expand(L, -1), w, "amin").view(L, S, S)
        out = torch.full((len(sources), L, S), inf, dtype=torch.float64, device=self.dev)
        for j, s in enumerate(sources):
            dist = out[j]
            dist[:, int(s)] = 0.0
            while True:
                new = torch.minimum(dist, (dist[:, :, None] + W).amin(1))
                if torch.equal(new, dist):
                    break
                dist = new
            out[j] = dist
        return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "parcel"):
        return None          # the batch carries its step sizes from round to round; the sweep is a long sequence
    e = _Exact(_problem(case["species"], case["layers"], seed, case.get("bins", 1000), case.get("diffuse", 0)))
    n = e.t(e.p.f0) * e.ng
    if case.get("start") == "equilibrium":
        n = e.equilibrium(n) * e.ng
    if kind == "steps":
        return e.steps(n, case["dt0"], case["steps"])
    if kind == "delta":
        return e.delta(n, case["dt"])
    if kind == "photolysis":
        return e.photolysis(n)
    if kind == "equilibrium":
        return e.equilibrium(n)
    wf, wb, _ = e.terms(n)
    q = torch.stack([wf, wb], -1)
    sources = 2 + np.random.default_rng([seed, 7]).choice(case["species"] - 2, size=case["sources"], replace=False)
    return dict(q=q, dist=e.distances(q, sources), pred_sp=None, pred_edge=None, lim_edge=None, lim_w=None)
