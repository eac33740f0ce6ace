"""The work that a user of this framework has it do, as cases that can be
timed: one call (or the few calls that belong together) of the public
interface each, on systems of the sizes that the workloads, the tests and the
benchmark have.

  listed()             the cases themselves
  draw(rng)            one more case from the same ranges
  prepare(case, seed)  what a program holds before the call, on the GPU
  run(state)           one pass; returns all that the call computes
  work(case)           the bytes and operations one pass cannot do without
  exact(case, seed)    what run() returns, from plain FP64 torch

A case names a system and an operation ("op"):

  orth_free     roks_orthonormalize_noalloc of a block (S = 1)
  orth          roks_orthonormalize of orbitals that a step has moved
  density       roks_density, then roks_potential with its energies
  apply         roks_apply_h: F|n>, S|n> and the gradient at fixed potentials
  precondition  roks_precondition of a residual block, with the network or not
  forces        roks_forces on orbitals written into a buffer
  pcg           one roks_pcg_step from orbitals written into a buffer
  diis          one roks_diis_step from orbitals written into a buffer
  train         one Adam step of the preconditioner network

The orbitals are seeded, damped plane-wave coefficients, S-orthonormalised
here: bands of rising kinetic energy, as in a run.  Real outputs that only a
mixed-precision call's FP64 interface widens are returned in FP32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_28637_gb300 import roks, synthetic as syn

TWO_PI = 2.0 * math.pi
GRIDS = (16, 24, 32, 48, 72, 96, 120)
# f_k^{sigma L} of the classes closed, a, b in up M, down M, up T, down T
F_TABLE = ((1.0, 1.0, 1.0, 1.0), (1.0, 0.0, 1.0, 0.0), (0.0, 1.0, 1.0, 0.0))
ENERGIES = ("E_kin", "E_loc", "E_nl", "E_H", "E_x_M", "E_x_T", "E_M", "E_T", "E_total")
# the largest listed system bounds what a drawn case may cost
MAX_BANDS, MAX_GRID = 430, 120


# ---------------------------------------------------------------- cases
def listed() -> list:
    return [
        # the smallest call: a solver loop inside another framework orthonormalises a few bands
        {"name": "orth_free 6 bands fp64", "op": "orth_free", "precision": "fp64", "npw": 1045, "bands": 6},
        # one step on the small systems that the network is trained on: launches and latency
        {"name": "pcg tiny-16 fp64", "op": "pcg", "system": "tiny-16", "precision": "fp64"},
        # a molecule's step in the solver, mixed precision
        {"name": "pcg organic-96 mixed", "op": "pcg", "system": "organic-96", "precision": "mixed"},
        # density and potentials of a molecule with the functional the paper computes molecules with
        {"name": "density organic-96 pbe mixed", "op": "density", "system": "organic-96", "precision": "mixed",
         "xc": "pbe_x"},
        # the FP64 path's apply on a molecule
        {"name": "apply organic-96 fp64", "op": "apply", "system": "organic-96", "precision": "fp64"},
        # the learned preconditioner on a molecule's residual
        {"name": "precondition organic-96 net", "op": "precondition", "system": "organic-96", "precision": "mixed",
         "network": True},
        # a training step of that network, on the pairs of some small systems
        {"name": "train 100001 samples", "op": "train", "samples": 100001},
        # orthonormalisation of a hundred bands in a solid
        {"name": "orth mgo-72 mixed", "op": "orth", "system": "mgo-72", "precision": "mixed"},
        # the apply on real orbitals at the Gamma point in a solid
        {"name": "apply mgo-72 gamma mixed", "op": "apply", "system": "mgo-72", "precision": "mixed", "gamma": 1},
        # the benchmark's system: the apply with its gradient
        {"name": "apply mgo-120 mixed", "op": "apply", "system": "mgo-120", "precision": "mixed"},
        # the benchmark's system: a whole solver step
        {"name": "diis mgo-120 mixed", "op": "diis", "system": "mgo-120", "precision": "mixed"},
        # the hybrid functional: an apply with all exchange pairs
        {"name": "apply hybrid-72 mixed", "op": "apply", "system": "hybrid-72", "precision": "mixed"},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng) -> dict:
    op = rng.choice(("orth_free", "orth", "density", "density", "apply", "apply", "apply", "precondition", "forces",
                     "pcg", "diis", "diis", "train"))
    if op == "train":
        return {"op": op, "samples": _log_int(rng, 3000, 400000)}
    precision = rng.choice(("mixed", "mixed", "mixed", "fp64"))
    if op == "orth_free":
        return {"op": op, "precision": precision, "npw": _log_int(rng, 500, 40000), "bands": _log_int(rng, 2, 64)}
    fp64 = precision == "fp64"
    grid = rng.choice(GRIDS[:5] if fp64 else GRIDS)
    # most spheres hold the density without aliasing (4 nmax < N); some are wider
    nmax = (grid - 1) // 4 if rng.random() < 0.8 else (grid - 1) * 2 // 5
    nmax = max(3, nmax - rng.randrange(0, 2 + nmax // 6))
    length = round(rng.uniform(0.8, 1.2) * (5.0 + 0.15 * grid), 3)
    npw = 4.0 * nmax ** 3
    most = int(min(MAX_BANDS if not fp64 else 96, npw / 8))
    if op == "pcg":
        most = min(most, 64)
    bands = _log_int(rng, 3, max(4, most))
    mode = rng.choice((0, 1, 1, 2))
    # an atom for each one to three bands, at most as dense as the solids
    atoms = max(1, min(215, round(bands * rng.uniform(0.3, 0.9)), int(length ** 3 / 60.0)))
    case = {"op": op, "system": "cell", "precision": precision, "grid": grid, "nmax": nmax, "L": length,
            "atoms": atoms, "closed": max(1, bands - (2 if mode else 0)), "mode": mode}
    if op == "apply" and not fp64 and bands <= 40 and grid <= 72 and rng.random() < 0.3:
        case["alpha"] = 0.25
    elif op in ("apply", "density", "orth") and rng.random() < 0.25:
        case["gamma"] = 1
        if mode and case["closed"] % 2:
            case["closed"] += 1
    elif op == "apply" and rng.random() < 0.2:
        case["empty"] = rng.randrange(1, 5)
    if op in ("density", "pcg", "diis") and rng.random() < 0.4:
        case["xc"] = "pbe_x"
    if op == "precondition":
        case["network"] = rng.random() < 0.6
    return case


# ---------------------------------------------------------------- systems
def _config(case: dict, seed: int) -> dict:
    """The system's description (synthetic.make_config's form)."""
    if case["system"] != "cell":
        cfg = syn.make_config(case["system"], seed % 100003)
        cfg = syn.with_changes(cfg, mode=case.get("mode", cfg["mode"]))
    else:
        r = np.random.default_rng([seed, 17])
        L, na = case["L"], case["atoms"]
        # atoms on a jittered lattice; every other one heavy (two radii), as in the molecules
        side = math.ceil(na ** (1.0 / 3.0))
        at = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:na]
        pos = ((at + 0.5 + r.uniform(-0.2, 0.2, (na, 3))) * (L / side)) % L
        species = []
        for radii in ((0.8,), (0.8, 1.2)):
            l = [0] * len(radii) + [1] * (3 * len(radii))
            m = [0] * len(radii) + [0, 1, 2] * len(radii)
            rc = list(radii) + [x for x in radii for _ in range(3)]
            D, Q = r.uniform(-0.5, 0.5, (len(l), len(l))), r.uniform(-1.0, 1.0, (len(l), len(l)))
            species.append({"l": l, "m": m, "rc": rc, "D": 0.5 * (D + D.T), "Q": 0.025 * (Q + Q.T)})
        atoms = [{"pos": tuple(map(float, p)), "species": i % 2, "depth": float(r.uniform(1.0, 3.0)), "width": 1.0}
                 for i, p in enumerate(pos)]
        cfg = {"name": "cell", "L": float(L), "grid": case["grid"],
               "ecut": 0.5 * (TWO_PI / L * (case["nmax"] + 0.3)) ** 2, "atoms": atoms, "species": species,
               "n_closed": case["closed"], "mode": case["mode"], "alpha": case.get("alpha", 0.0), "seed": seed % 100003}
    if "empty" in case:
        cfg["n_empty"] = case["empty"]
    cfg["xc"] = case.get("xc", "slater")
    return cfg


def _sizes(case: dict) -> dict:
    """Counts of a case's system, for work()."""
    cfg = _config(case, 0)
    q = cfg["L"] / TWO_PI
    M = int(math.floor(2.0 * cfg["ecut"] * q * q))
    n = math.isqrt(M)
    i = np.arange(-n, n + 1)
    ij = i[:, None] ** 2 + i[None, :] ** 2
    kmax = np.floor(np.sqrt(np.maximum(M - ij, 0)) + 1e-9)
    inside = ij <= M
    npw = int((2 * kmax[inside] + 1).sum())
    nb = syn.n_bands(cfg)
    return {"N": cfg["grid"], "npw": (npw + 1) // 2 if case.get("gamma") else npw, "ncol": int(inside.sum()),
            "np": 2 * n + 1, "nb": nb, "transforms": (nb + 1) // 2 if case.get("gamma") else nb,
            "nproj": sum(len(cfg["species"][a["species"]]["l"]) for a in cfg["atoms"]), "natoms": len(cfg["atoms"]),
            "cs": 16 if case["precision"] == "fp64" else 8}


class _Model:
    """The model system in plain torch: FP64 for exact(); its plane waves,
    projectors and overlap (in the element type) make the inputs as well."""

    def __init__(self, cfg: dict, dtype=torch.complex128, gamma: bool = False, device: str = "cuda"):
        self.cfg, self.cdt, self.dev, self.gamma = cfg, dtype, device, gamma
        self.L, self.N, self.omega = cfg["L"], cfg["grid"], cfg["L"] ** 3
        self.mode, self.nc = cfg["mode"], cfg["n_closed"]
        self.nocc = self.nc + (0 if self.mode == 0 else 2)
        self.nb = syn.n_bands(cfg)
        self.alpha = cfg.get("alpha", 0.0)
        q = self.L / TWO_PI
        M = int(math.floor(2.0 * cfg["ecut"] * q * q))
        n = math.isqrt(M)
        i = torch.arange(-n, n + 1, device=device)
        m = torch.stack(torch.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3)
        self.miller = m[(m * m).sum(1) <= M]
        self.npw = self.miller.shape[0]
        self.h0 = (self.npw - 1) // 2
        self.rows = self.npw - self.h0 if gamma else self.npw
        self.G = self.miller.double() * (TWO_PI / self.L)
        self.g2 = (self.G ** 2).sum(1)
        w = self.miller % self.N
        self.gidx = (w[:, 0] * self.N + w[:, 1]) * self.N + w[:, 2]
        self.P, self.D, self.Q = self._projectors()
        f = torch.tensor(F_TABLE, dtype=torch.float64, device=device)
        cM, cT = {0: (1.0, 0.0), 1: (2.0, -1.0), 2: (0.0, 1.0)}[self.mode]
        self.cM, self.cT = cM, cT
        cch = torch.tensor([cM, cM, cT, cT], dtype=torch.float64, device=device)
        self.f, self.C = f, f * cch
        self.w = self.C.sum(1)
        self.wx = (f * cch) @ f.T
        self.cls = torch.tensor([0] * self.nc + [1, 2] * (self.mode != 0) + [0] * (self.nb - self.nocc), device=device)

    def _projectors(self):
        cfg = self.cfg
        na = len(cfg["atoms"])
        offs, n = [], 0
        for a in cfg["atoms"]:
            offs.append(n)
            n += len(cfg["species"][a["species"]]["l"])
        P = torch.zeros((self.npw, n), dtype=self.cdt, device=self.dev)
        D = torch.zeros((n, n), dtype=torch.float64)
        Q = torch.zeros((n, n), dtype=torch.float64)
        self.owner = torch.zeros(n, dtype=torch.long)
        pos = torch.tensor([a["pos"] for a in cfg["atoms"]], dtype=torch.float64, device=self.dev).reshape(na, 3)
        for s, sp in enumerate(cfg["species"]):
            mine = [a for a in range(na) if cfg["atoms"][a]["species"] == s]
            if not mine:
                continue
            ph = -(self.G @ pos[mine].T)
            ph = torch.complex(torch.cos(ph), torch.sin(ph))
            for c, (l, mm, rc) in enumerate(zip(sp["l"], sp["m"], sp["rc"])):
                norm = (math.pi * rc * rc) ** -0.75 * (math.sqrt(2.0 / (rc * rc)) if l == 1 else 1.0)
                rad = norm * (TWO_PI * rc * rc) ** 1.5 / math.sqrt(self.omega) * torch.exp(-0.5 * self.g2 * rc * rc)
                ang = (-1j * rc * rc) * self.G[:, mm] if l == 1 else torch.ones_like(self.g2)
                P[:, [offs[a] + c for a in mine]] = ((rad * ang)[:, None] * ph).to(self.cdt)
            k = len(sp["l"])
            for a in mine:
                sl = slice(offs[a], offs[a] + k)
                D[sl, sl] = torch.as_tensor(np.asarray(sp["D"]).reshape(k, k))
                Q[sl, sl] = torch.as_tensor(np.asarray(sp["Q"]).reshape(k, k))
                self.owner[sl] = a
        return P, D.to(self.dev), Q.to(self.dev)

    # ------------------------------------------------ stored form of real orbitals (Gamma)
    def expand(self, psi):
        """Full-sphere columns of the stored half-sphere ones."""
        if not self.gamma:
            return psi
        c = psi / math.sqrt(2.0)
        c[0] = psi[0]
        return torch.cat([torch.flip(c[1:], [0]).conj(), c])

    def restrict(self, full):
        if not self.gamma:
            return full
        c = full[self.h0:] * math.sqrt(2.0)
        c[0] = full[self.h0]
        return c

    # ------------------------------------------------ overlap
    def overlap(self, psi):
        B = self.P.conj().T @ psi
        O = psi.conj().T @ psi + B.conj().T @ (self.Q.to(B.dtype) @ B)
        return 0.5 * (O + O.conj().T)

    def orthonormalize(self, psi):
        L = torch.linalg.cholesky(self.overlap(psi).to(torch.complex128))
        X = torch.linalg.solve_triangular(L, torch.eye(L.shape[0], dtype=L.dtype, device=L.device), upper=False)
        return psi @ X.conj().T.to(psi.dtype)

    # ------------------------------------------------ grid
    def to_real(self, c):
        """psi(r) of columns c, as rows of N^3 points."""
        g = torch.zeros((c.shape[1], self.N ** 3), dtype=torch.complex128, device=self.dev)
        g[:, self.gidx] = c.T
        r = torch.fft.ifftn(g.reshape(-1, self.N, self.N, self.N), dim=(1, 2, 3), norm="forward")
        return r.reshape(c.shape[1], -1) / math.sqrt(self.omega)

    def to_pw(self, f):
        F = torch.fft.fftn(f.reshape(-1, self.N, self.N, self.N), dim=(1, 2, 3)).reshape(f.shape[0], -1)
        return (F[:, self.gidx] * (math.sqrt(self.omega) / self.N ** 3)).T

    def blocks(self, n: int):
        step = max(1, int(4e7 / self.N ** 3))
        return [slice(i, min(n, i + step)) for i in range(0, n, step)]

    def frequencies(self):
        t = torch.arange(self.N, device=self.dev)
        return torch.where(t <= self.N // 2, t, t - self.N).double() * (TWO_PI / self.L)

    def grid_g2(self):
        g = self.frequencies() ** 2
        return (g[:, None, None] + g[None, :, None] + g[None, None, :]).reshape(-1)

    def _grid(self, f, inverse):
        f = f.to(torch.complex128).reshape(-1, self.N, self.N, self.N)
        fn = torch.fft.ifftn if inverse else torch.fft.fftn
        return fn(f, dim=(1, 2, 3), norm="forward").reshape(f.shape[0], -1)

    def wells(self, only=None):
        """V(G) of the local wells (Nyquist planes left out), or of one atom's."""
        N, g = self.N, self.frequencies()
        g2 = self.grid_g2()
        out = torch.zeros(N ** 3, dtype=torch.complex128, device=self.dev)
        for a, at in enumerate(self.cfg["atoms"]):
            if only is not None and a != only:
                continue
            ph = [torch.exp(-1j * g * x) for x in at["pos"]]
            sf = (ph[0][:, None, None] * ph[1][None, :, None] * ph[2][None, None, :]).reshape(-1)
            out += -(at["depth"] * (TWO_PI * at["width"] ** 2) ** 1.5 / self.omega) * torch.exp(
                -0.5 * g2 * at["width"] ** 2) * sf
        keep = torch.ones(N, dtype=torch.bool, device=self.dev)
        keep[N // 2] = False
        return out * (keep[:, None, None] & keep[None, :, None] & keep[None, None, :]).reshape(-1)

    # ------------------------------------------------ densities, potentials, energies
    def densities(self, psi):
        rho = torch.zeros((3, self.N ** 3), dtype=torch.float64, device=self.dev)
        for s in self.blocks(self.nocc):
            r = self.to_real(psi[:, s])
            d = r.real ** 2 + r.imag ** 2
            for k in range(3):
                rho[k] += d[self.cls[s] == k].sum(0)
        return rho

    def _derivative(self, f, axis):
        g = self.frequencies()
        g[self.N // 2] = 0.0
        shape = [1, 1, 1]
        shape[axis] = self.N
        mult = g.reshape(shape).expand(self.N, self.N, self.N).reshape(-1)
        return self._grid(1j * mult * self._grid(f, False)[0], True)[0].real

    def _exchange_channels(self, rho_ch):
        r = rho_ch.clamp(min=0.0)
        c = r ** (1.0 / 3.0)
        c6 = (6.0 / math.pi) ** (1.0 / 3.0)
        cx, dv, scale = 0.75 * c6, self.omega / self.N ** 3, 1.0 - self.alpha
        if self.cfg.get("xc", "slater") == "slater":
            return -scale * c6 * c, -scale * cx * dv * (c * r).sum(1)
        k2, kappa, mu = (6.0 * math.pi ** 2) ** (2.0 / 3.0), 0.804, 0.06672455060314922 * math.pi ** 2 / 3.0
        v, e = torch.zeros_like(r), torch.zeros(4, dtype=torch.float64, device=self.dev)
        for ch in range(4):
            grad = [self._derivative(r[ch], a) for a in range(3)]
            on = r[ch] > 1e-10
            rr = torch.where(on, r[ch], torch.ones_like(r[ch]))
            cc = rr ** (1.0 / 3.0)
            s2 = torch.where(on, sum(x * x for x in grad) / (4.0 * k2 * rr ** 2 * cc ** 2), torch.zeros_like(rr))
            den = 1.0 + mu * s2 / kappa
            F, dF = 1.0 + mu * s2 / den, mu / (den * den)
            zero = torch.zeros_like(rr)
            v1 = torch.where(on, -(4.0 / 3.0) * cx * cc * (F - 2.0 * s2 * dF), zero)
            fl = torch.where(on, -cx * dF / (2.0 * k2 * rr * cc), zero)
            v[ch] = scale * (v1 - sum(self._derivative(fl * grad[a], a) for a in range(3)))
            e[ch] = scale * dv * torch.where(on, -cx * rr * cc * F, zero).sum()
        return v, e

    def potentials(self, rho):
        rho_ch = self.f.T @ rho
        tot = rho_ch[0] + rho_ch[1]
        g2 = self.grid_g2()
        rG = self._grid(tot, False)[0]
        k = torch.where(g2 > 0, 4.0 * math.pi / g2.clamp(min=1e-300), torch.zeros_like(g2))
        vh = self._grid(k * rG, True)[0].real
        vloc = self._grid(self.wells(), True)[0].real
        vx, ex = self._exchange_channels(rho_ch)
        V = self.w[:, None] * (vloc + vh) + self.C @ vx
        dv = self.omega / self.N ** 3
        E = {"E_H": 0.5 * self.omega * float((k * rG.abs() ** 2).sum()), "E_loc": dv * float((vloc * tot).sum()),
             "E_x_M": float(ex[0] + ex[1]), "E_x_T": float(ex[2] + ex[3])}
        return V, E

    def energies(self, psi, E):
        psi = psi[:, :self.nocc]
        w = self.w[self.cls[:self.nocc]]
        B = self.P.conj().T @ psi
        E = dict(E)
        E["E_kin"] = float((w * (0.5 * self.g2[:, None] * psi.abs() ** 2).sum(0)).sum())
        E["E_nl"] = float((w * (B.conj() * (self.D.to(B.dtype) @ B)).real.sum(0)).sum())
        one = E["E_kin"] + E["E_loc"] + E["E_nl"] + E["E_H"]
        E["E_M"], E["E_T"] = one + E["E_x_M"], one + E["E_x_T"]
        E["E_total"] = self.cM * E["E_M"] + self.cT * E["E_T"]
        return {k: E[k] for k in ENERGIES}

    def energy(self, psi):
        return self.energies(psi, self.potentials(self.densities(psi))[1])["E_total"]

    # ------------------------------------------------ operators
    def apply(self, psi, V, cls=None):
        cls = self.cls if cls is None else cls
        w = self.w[cls]
        F = torch.empty_like(psi)
        for s in self.blocks(psi.shape[1]):
            F[:, s] = self.to_pw(V[cls[s]] * self.to_real(psi[:, s]))
        B = self.P.conj().T @ psi
        F += 0.5 * w * self.g2[:, None] * psi + self.P @ (w * (self.D.to(B.dtype) @ B))
        if self.alpha:
            F += self._exact_exchange(psi, cls)
        return F, psi + self.P @ (self.Q.to(B.dtype) @ B)

    def _exact_exchange(self, psi, cls):
        g2 = self.grid_g2()
        Rc = (3.0 * self.omega / (4.0 * math.pi)) ** (1.0 / 3.0)
        v = torch.where(g2 > 0, 4.0 * math.pi * (1.0 - torch.cos(g2.sqrt() * Rc)) / g2.clamp(min=1e-300),
                        torch.full_like(g2, TWO_PI * Rc * Rc))
        r = self.to_real(psi)
        out = torch.empty_like(psi)
        for n in range(psi.shape[1]):
            X = torch.zeros(self.N ** 3, dtype=torch.complex128, device=self.dev)
            for s in self.blocks(psi.shape[1]):
                W = self._grid(v * self._grid(r[s].conj() * r[n], False), True)
                X += (self.wx[cls[n], self.cls[s]][:, None] * r[s] * W).sum(0)
            out[:, n] = -self.alpha * self.to_pw(X[None])[:, 0]
        return out

    def tpa(self, g):
        a2 = g.abs() ** 2
        X = 1.5 * (self.g2[:, None] * a2).sum(0) / a2.sum(0).clamp(min=1e-300)
        x = self.g2[:, None] / X
        num = 27.0 + x * (18.0 + x * (12.0 + 8.0 * x))
        return -(2.0 / X) * num / (num + 16.0 * x ** 4)


def _uniform(gen, *shape, dtype):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=dtype) * 2.0 - 1.0


def _random_block(m: _Model, seed: int, stream: int, bands: int, power) -> torch.Tensor:
    """Damped coefficients c_G = u / (1 + |G|^2)^power of the stored rows."""
    gen = torch.Generator("cuda").manual_seed(seed * 1000003 + stream)
    rdt = torch.float64 if m.cdt == torch.complex128 else torch.float32
    u = _uniform(gen, m.rows, bands, 2, dtype=rdt)
    g2 = (m.g2[m.h0:] if m.gamma else m.g2).to(rdt)
    u = torch.view_as_complex(u) * (1.0 + g2)[:, None] ** -torch.as_tensor(power, dtype=rdt, device="cuda")
    if m.gamma:
        u[0] = u[0].real.to(u.dtype)
        u[1:] *= math.sqrt(2.0)
    return u


def _orbitals(m: _Model, seed: int) -> torch.Tensor:
    """S-orthonormal bands of rising kinetic energy (stored rows x bands)."""
    u = _random_block(m, seed, 1, m.nb, np.linspace(2.5, 1.0, m.nb))
    return m.restrict(m.orthonormalize(m.expand(u))).contiguous()


def _moved(m: _Model, seed: int, psi) -> torch.Tensor:
    """Orbitals that a step has moved: no longer orthonormal."""
    d = _random_block(m, seed, 2, m.nb, 1.0)
    return psi + 0.1 * d / d.abs().pow(2).sum(0).sqrt()


def _residual(m: _Model, seed: int) -> torch.Tensor:
    return _random_block(m, seed, 3, m.nb, np.linspace(0.7, 1.1, m.nb))


def _network(seed: int) -> np.ndarray:
    """Weights of a trained network's size and spread."""
    r = np.random.default_rng([seed, 5])
    p = syn.mlp_initial_params(seed % 100003) + r.normal(0.0, 0.05, syn.MLP_NPARAM)
    return p.astype(np.float32)


def _cdtype(case):
    return torch.complex128 if case["precision"] == "fp64" else torch.complex64


def _padded(cols, ld: int) -> torch.Tensor:
    """(rows x bands) columns as the library's (bands, ld) block."""
    out = torch.zeros((cols.shape[1], ld), dtype=cols.dtype, device="cuda")
    out[:, :cols.shape[0]] = cols.T
    return out


def _free_block(case, seed):
    """Bands that a step has moved away from orthonormal ones, S = 1."""
    gen = torch.Generator("cuda").manual_seed(seed * 1000003 + 7)
    n, nb = case["npw"], case["bands"]
    damp = 1.0 / (1.0 + 40.0 * torch.arange(n, device="cuda", dtype=torch.float64) / n)
    a = torch.view_as_complex(_uniform(gen, n, nb, 2, dtype=torch.float64)) * damp[:, None]
    a = torch.linalg.qr(a)[0]
    d = torch.view_as_complex(_uniform(gen, n, nb, 2, dtype=torch.float64)) * damp[:, None]
    return (a + 0.1 * d / d.abs().pow(2).sum(0).sqrt()).to(_cdtype(case))


def _train_data(case, seed):
    r = np.random.default_rng([seed, 11])
    n = case["samples"]
    band = r.integers(0, max(1, n // 1045), n)
    eps = r.uniform(-1.5, 1.0, band.max() + 1)[band]
    feats = np.stack([np.log1p(r.gamma(1.0, 1.0, n)), np.log1p(r.gamma(0.5, 1.0, n)), eps], 1)
    target = np.clip(0.8 * np.sin(2.0 * feats[:, 0]) - 0.5 * feats[:, 1] + 0.2 * eps + r.normal(0, 0.3, n), -3, 3)
    weight = r.gamma(0.5, 1.0, n) / 1045.0
    p = _network(seed)
    mom = r.normal(0.0, 1e-3, p.shape)
    var = (np.abs(r.normal(0.0, 3e-3, p.shape)) + 1e-3) ** 2
    return [torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
            for x in (feats, target, weight, p, mom, var)]


TRAIN = {"step": 12, "lr": 2e-3}
DIIS = {"history": 6, "tau": 0.5, "lambda_ab": 0.5, "lambda_ba": -0.5}


# ---------------------------------------------------------------- prepare, run
def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    st = {"case": case, "op": op}
    if op == "train":
        f, t, w, p, m, v = _train_data(case, seed)
        st.update(feats=f, target=t, weight=w, p0=p, m0=m, v0=v, p=p.clone(), m=m.clone(), v=v.clone(),
                  grad=torch.zeros_like(p), loss=torch.zeros(1, device="cuda"), n=case["samples"],
                  work=torch.empty(roks.roks_mlp_grad_work(case["samples"]), device="cuda"))
        return st
    if op == "orth_free":
        a = _free_block(case, seed)
        ld = (case["npw"] + 31) // 32 * 32
        st.update(psi0=_padded(a, ld), psi=_padded(a, ld), ld=ld,
                  prec=roks.ROKS_FP64 if case["precision"] == "fp64" else roks.ROKS_MIXED)
        return st
    cfg = _config(case, seed)
    m = _Model(cfg, _cdtype(case), bool(case.get("gamma")))
    psi = _orbitals(m, seed)
    ctx = roks.Context(cfg, case["precision"], gamma=case.get("gamma", 0), max_iter=0)
    st.update(ctx=ctx, ld=ctx.ld)
    if op == "orth":
        psi = _moved(m, seed, psi)
    st["psi0"] = _padded(psi, ctx.ld)
    st["psi"] = st["psi0"].clone()
    if op == "density":
        st["rho"] = (torch.empty((3, ctx.N ** 3), dtype=torch.float64, device="cuda")
                     if case["precision"] == "fp64" else None)
        st["V"] = torch.empty((3, ctx.N ** 3), dtype=ctx.rdtype, device="cuda")
    if op in ("apply", "precondition"):
        # the potentials of these orbitals, as an iteration has them before the apply
        ctx.density(st["psi"])
        ctx.potential()
        for k in ("F", "S", "g"):
            st[k] = ctx.new_bands()
    if op == "precondition":
        # theta of the orbitals gives the band energies that the network takes
        roks.roks_apply_h(ctx.ctx, st["psi"], ctx.ld, st["F"], st["S"], st["g"])
        st["res"] = _padded(_residual(m, seed), ctx.ld)
        st["out"] = st["F"]
        st["out"].zero_()
        del st["S"], st["g"]
        if case.get("network"):
            ctx.set_preconditioner(torch.from_numpy(_network(seed)).cuda())
    torch.cuda.synchronize()
    return st


def run(st: dict):
    op = st["op"]
    if op == "train":
        for k in ("p", "m", "v"):
            st[k].copy_(st[k + "0"])
        stream = torch.cuda.current_stream().cuda_stream
        roks.roks_mlp_grad(st["n"], st["feats"], st["target"], st["weight"], st["p"], st["work"], st["grad"],
                           st["loss"], stream)
        roks.roks_mlp_adam(st["p"], st["m"], st["v"], st["grad"], TRAIN["step"], TRAIN["lr"], stream=stream)
        return {k: st[k] for k in ("grad", "loss", "p", "m", "v")}
    st["psi"].copy_(st["psi0"])
    if op == "orth_free":
        c = st["case"]
        roks.roks_orthonormalize_noalloc(st["prec"], c["npw"], c["bands"], st["psi"], st["ld"],
                                         torch.cuda.current_stream().cuda_stream)
        return {"psi": st["psi"]}
    ctx = st["ctx"]
    if op == "orth":
        return {"psi": ctx.orthonormalize(st["psi"])}
    if op == "density":
        roks.roks_density(ctx.ctx, st["psi"], st["ld"], st["rho"])
        e = roks.roks_potential(ctx.ctx, st["V"])
        return {"rho": st["rho"], "V": st["V"], "E": {k: e[k] for k in ENERGIES}}
    if op == "apply":
        roks.roks_apply_h(ctx.ctx, st["psi"], st["ld"], st["F"], st["S"], st["g"])
        return {"F": st["F"], "S": st["S"], "g": st["g"]}
    if op == "precondition":
        roks.roks_precondition(ctx.ctx, st["res"], st["ld"], st["out"])
        return {"out": st["out"]}
    ctx.invalidate()
    if op == "forces":
        F = ctx.forces(st["psi"])
        return {"F": F if st["case"]["precision"] == "fp64" else F.astype(np.float32)}
    if op == "diis":
        i = ctx.diis_step(st["psi"], **DIIS)
        return {"psi": st["psi"], "E": i["E"], "E_new": i["E_new"], "residual": i["res_norm"]}
    i = ctx.pcg_step(st["psi"])
    return {"psi": st["psi"], "E": i["E"], "E_new": i["E_new"], "step": i["step"], "gradient": i["grad_norm"]}


# ---------------------------------------------------------------- work
def work(case: dict) -> dict:
    op = case["op"]
    if op == "train":
        n, H = case["samples"], syn.MLP_HIDDEN
        # forward, back-propagation through both layers, and the weight gradients
        return {"bytes": 4.0 * (5 * n + 7 * syn.MLP_NPARAM), "flops": 2.0 * n * (3 * (H * H + H) + 2 * 3 * H)}
    cs = 16 if case["precision"] == "fp64" else 8
    if op == "orth_free":
        n, nb = case["npw"], case["bands"]
        return {"bytes": 2.0 * cs * n * nb, "flops": 8.0 * n * nb * nb + 4.0 * nb ** 3}
    s = _sizes(case)
    N, npw, nb, nproj, nt = s["N"], s["npw"], s["nb"], s["nproj"], s["transforms"]
    N3, block = float(N) ** 3, float(cs) * s["npw"] * nb
    # one direction of all bands' transforms, sphere columns and planes only
    fft = 5.0 * nt * N * math.log2(N) * (s["ncol"] + s["np"] * N + N * N)
    band2, proj = 8.0 * npw * nb * nb, 8.0 * npw * nproj * nb
    rs = cs // 2
    P = float(cs) * npw * nproj
    if case.get("gamma"):
        band2, proj = band2 / 2, proj / 2
    grid = 5.0 * N3 * math.log2(N3)   # one complex grid transform
    apply_f = 2 * fft + 8.0 * nt * N3 / 4 + 2 * proj   # P^H psi, P (D B)
    if case.get("alpha") or case.get("system") == "hybrid-72":
        apply_f += nb * (nb + 1) / 2.0 * (2 * grid + 30.0 * N3)
    dens_f = fft + 3.0 * nt * N3 + proj + 2 * grid + (16 * grid if case.get("xc") == "pbe_x" else 0.0)
    orth_f = band2 + proj + 8.0 * nproj * nb * nb + 4.0 * nb ** 3 + band2
    if op == "orth":
        return {"bytes": 2 * block + P, "flops": orth_f}
    if op == "density":
        return {"bytes": block + P + rs * 5 * N3, "flops": dens_f}
    if op == "apply":
        return {"bytes": 4 * block + P + rs * 3 * N3, "flops": apply_f + proj + 2 * band2}
    if op == "precondition":
        H = syn.MLP_HIDDEN
        return {"bytes": 2 * block, "flops": float(npw) * nb * (2.0 * (H * H + 4 * H) if case.get("network") else 20.0)}
    if op == "forces":
        return {"bytes": block + P + rs * 3 * N3, "flops": dens_f + apply_f + band2 + 3 * proj + 20.0 * s["natoms"] * N3}
    if op == "diis":
        return {"bytes": 2 * block + P, "flops": 2 * dens_f + apply_f + 2 * band2 + orth_f}
    return {"bytes": 2 * block + P,
            "flops": 3 * dens_f + apply_f + proj + 5 * band2 + 2 * (orth_f + band2 + 20.0 * nb ** 3)}


# ---------------------------------------------------------------- exact
def _expm(A):
    return torch.linalg.matrix_exp(A)


def _gradient(m: _Model, psi, F, S):
    th = psi.conj().T @ F
    th[:, m.nocc:] = 0.0
    F = F.clone()
    F[:, m.nocc:] = 0.0
    return F - S @ (0.5 * (th + th.conj().T))


def _exact_forces(m: _Model, psi) -> np.ndarray:
    rho = m.densities(psi)
    F, _ = m.apply(psi, m.potentials(rho)[0])
    th = psi.conj().T @ F
    gam = 0.5 * (th + th.conj().T)
    rG = m._grid((m.w[:, None] * rho).sum(0), False)[0].conj()
    g = m.frequencies()
    N = m.N
    axes = [g[:, None, None], g[None, :, None], g[None, None, :]]
    out = torch.zeros((len(m.cfg["atoms"]), 3), dtype=torch.float64, device=m.dev)
    for a in range(len(m.cfg["atoms"])):
        v = (m.wells(a) * rG).reshape(N, N, N)
        for nu in range(3):
            out[a, nu] = (-1j * axes[nu] * v).sum().real * m.omega
    B = m.P.conj().T @ psi
    w = m.w[m.cls]
    Y = w * (m.D.to(B.dtype) @ B) - (m.Q.to(B.dtype) @ B) @ gam
    own = m.owner.to(m.dev)
    for nu in range(3):
        dB = (-1j * m.G[:, nu][:, None] * m.P).conj().T @ psi
        out[:, nu].index_add_(0, own, 2.0 * (dB.conj() * Y).real.sum(1))
    return -out.cpu().numpy()


def _exact_pcg(m: _Model, psi):
    V, E = m.potentials(m.densities(psi))
    E0 = m.energies(psi, E)["E_total"]
    F, S = m.apply(psi, V)
    th = psi.conj().T @ F
    G = F - S @ (0.5 * (th + th.conj().T))
    gI, gin = F - S @ th, th - th.conj().T
    pI = m.tpa(gI) * gI
    pI = pI - psi @ (S.conj().T @ pI)
    # <m|F^c|m>: the closed bands have it in theta
    d = th.diagonal().real.clone()
    if m.mode:
        o = psi[:, m.nc:]
        Fc, _ = m.apply(o, V, torch.zeros(2, dtype=torch.long, device=m.dev))
        d[m.nc:] = (o.conj() * Fc).real.sum(0)
    shell = m.cls.clamp(max=1) if m.mode == 2 else m.cls
    lt = shell[:, None] < shell[None, :]
    R = torch.where(shell[:, None] == shell[None, :], th, torch.where(lt, th.conj().T - th, gin))
    r = R.abs()
    dd = d[:, None] - d[None, :]
    phi = -0.5 * torch.atan2(2.0 * r, dd.abs()) * torch.where(dd >= 0, 1.0, -1.0)
    A = torch.where(r >= 1e-14, phi * R / r.clamp(min=1e-300), torch.zeros_like(R)).triu(1)
    A = A - A.conj().T
    dE = 2.0 * float((pI.conj() * G).real.sum()) + float((A.conj() * gin).real.sum())
    if dE >= 0.0:
        A = torch.zeros_like(A)
        dE = 2.0 * float((pI.conj() * G).real.sum())

    def trial(t):
        return m.orthonormalize((psi + t * pI) @ _expm(t * A))

    dt = 0.3
    c = (m.energy(trial(dt)) - E0 - dE * dt) / (dt * dt)
    step = min(-dE / (2.0 * c) if c > 0.0 else dt, 3.0 * dt)
    new = trial(step)
    return new, E0, m.energy(new), step, float(torch.linalg.norm(G))


def _exact_diis(m: _Model, psi):
    V, E = m.potentials(m.densities(psi))
    E0 = m.energies(psi, E)["E_total"]
    F, S = m.apply(psi, V)
    th = psi.conj().T @ F
    lam = torch.full((m.nb, m.nb), 0.5, dtype=torch.float64, device=m.dev)
    if m.mode == 1:
        lam[m.nc, m.nc + 1], lam[m.nc + 1, m.nc] = DIIS["lambda_ab"], DIIS["lambda_ba"]
    R = F - S @ (th - lam * (th - th.conj().T))
    new = m.orthonormalize(psi + DIIS["tau"] * m.tpa(R) * R)
    return new, E0, m.energy(new), float(torch.linalg.norm(R))


def _evaluate(p, feats):
    """Network outputs for feature rows (FP64)."""
    H, o, parts = syn.MLP_HIDDEN, 0, []
    for shape in ((H, 3), (H,), (H, H), (H,), (H,), (1,)):
        n = math.prod(shape)
        parts.append(p[o:o + n].reshape(shape))
        o += n
    W1, b1, W2, b2, w3, b3 = parts
    return torch.tanh(torch.tanh(feats @ W1.T + b1) @ W2.T + b2) @ w3 + b3


def _exact_train(case, seed):
    f, t, w, p, mo, v = (x.double() for x in _train_data(case, seed))
    p.requires_grad_(True)
    loss = (w * (_evaluate(p, f) - t) ** 2).sum() / w.sum()
    loss.backward()
    g = p.grad
    b1, b2, eps, k = 0.9, 0.999, 1e-8, TRAIN["step"]
    mo, v = b1 * mo + (1 - b1) * g, b2 * v + (1 - b2) * g * g
    new = p.detach() - TRAIN["lr"] * (mo / (1 - b1 ** k)) / ((v / (1 - b2 ** k)).sqrt() + eps)
    return {"grad": g, "loss": loss.detach().reshape(1), "p": new, "m": mo, "v": v}


def exact(case: dict, seed: int):
    op = case["op"]
    if op == "train":
        return _exact_train(case, seed)
    if op == "orth_free":
        a = _free_block(case, seed).to(torch.complex128)
        L = torch.linalg.cholesky(a.conj().T @ a)
        X = torch.linalg.solve_triangular(L, torch.eye(L.shape[0], dtype=L.dtype, device="cuda"), upper=False)
        return {"psi": _padded(a @ X.conj().T, (case["npw"] + 31) // 32 * 32)}
    cfg, gamma = _config(case, seed), bool(case.get("gamma"))
    m = _Model(cfg, _cdtype(case), gamma)
    psi = _orbitals(m, seed)
    if op == "orth":
        psi = _moved(m, seed, psi)
    res = _residual(m, seed).to(torch.complex128) if op == "precondition" else None
    m = _Model(cfg, torch.complex128, gamma)
    psi = m.expand(psi.to(torch.complex128))
    ld = (m.rows + 31) // 32 * 32
    out = lambda cols: _padded(m.restrict(cols), ld)  # noqa: E731
    if op == "orth":
        return {"psi": out(m.orthonormalize(psi))}
    if op == "forces":
        F = _exact_forces(m, psi)
        return {"F": F if case["precision"] == "fp64" else F.astype(np.float32)}
    if op == "pcg":
        new, E0, E1, step, gn = _exact_pcg(m, psi)
        return {"psi": out(new), "E": E0, "E_new": E1, "step": step, "gradient": gn}
    if op == "diis":
        new, E0, E1, rn = _exact_diis(m, psi)
        return {"psi": out(new), "E": E0, "E_new": E1, "residual": rn}
    rho = m.densities(psi)
    V, E = m.potentials(rho)
    if op == "density":
        return {"rho": rho if case["precision"] == "fp64" else None, "V": V, "E": m.energies(psi, E)}
    F, S = m.apply(psi, V)
    if op == "apply":
        return {"F": out(F), "S": out(S), "g": out(_gradient(m, psi, F, S))}
    K = m.tpa(res)
    if case.get("network"):
        a2 = res.abs() ** 2
        T = (0.5 * m.g2[:, None] * a2).sum(0) / a2.sum(0)
        eps = (psi.conj() * F).sum(0).real / m.w[m.cls]
        p = torch.from_numpy(_network(seed)).cuda().to(torch.bfloat16).double()
        for n in range(m.nb):
            u = torch.stack([torch.log1p(0.5 * m.g2 / T[n]), torch.log1p((a2[:, n] / a2[:, n].mean()).sqrt()),
                             eps[n].expand(m.npw)], 1)
            K[:, n] *= torch.exp(_evaluate(p, u).clamp(-3.0, 3.0))
    return {"out": _padded(K * res, ld)}
