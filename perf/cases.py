"""Workloads whose speed is measured: variational Monte Carlo sweeps, wave-function and local-energy evaluations,
adjoint forces, stochastic reconfiguration and lattice-regularised DMC of JAGP wave functions, each one call (or the few
calls that belong together) of ``paper_2002_07401_gb300`` on device-resident walkers.

Systems are clusters of atoms at the density of the repository's 16-atom workload with s/p/d Gaussians, a random dense or
banded pairing matrix and one electron pair per atom (or a few unpaired electrons), drawn from the seed; walkers start
near the atoms.  ``exact`` restates the method in plain float64 torch.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2002_07401_gb300 as pg

# s, p, d shells per atom for so many functions' recipe (the repository's)
RECIPES = {6: (3, 1, 0), 16: (5, 2, 1), 20: (4, 2, 2), 24: (5, 3, 2)}
NCOMP = (1, 3, 5)
LRDMC_A, LRDMC_TAU, SR_ITERS = 0.2, 0.005, 50


def listed():
    base = {"prec": "fp64", "slater": False, "band": False, "refresh": 0, "tune": False, "unpaired": 0, "systems": 1}
    return [
        # the smallest runs (a molecule of four H, a few hundred walkers): launches and latency are all there is
        dict(base, name="sweep_h4_fp64", kind="sweep", atoms=4, recipe=6, walkers=256),
        # the plain FP64 sweep at its usual size (16 He, 32 electrons)
        dict(base, name="sweep_he16_fp64", kind="sweep", atoms=16, recipe=20, walkers=4096, tune=True),
        # the same with FP64-equivalent lambda products on the tensor cores
        dict(base, name="sweep_he16_fp64tc", kind="sweep", atoms=16, recipe=20, walkers=2048, prec="fp64tc"),
        # the production sweep: mixed precision
        dict(base, name="sweep_he16_mixed", kind="sweep", atoms=16, recipe=20, walkers=4096, prec="mixed", tune=True),
        # a larger, spin-polarised molecule of odd sizes with the inverse refreshed every 16 moves
        dict(base, name="sweep_odd43_mixed", kind="sweep", atoms=42, recipe=16, walkers=509, prec="mixed", refresh=16,
             unpaired=3),
        # the largest system: 256 He, 512 electrons, banded pairing matrix
        dict(base, name="sweep_he256_mixed", kind="sweep", atoms=256, recipe=16, walkers=64, prec="mixed", band=True),
        # many independent uneven molecules swept together (one graph replay per sweep)
        dict(base, name="batch_uneven_mixed", kind="batch", atoms=64, recipe=16, walkers=96, prec="mixed", refresh=16,
             systems=10),
        # log|Psi| and local energies of configurations that come from elsewhere, with Slater shells among the basis
        dict(base, name="energy_odd23_mixed", kind="energy", atoms=23, recipe=20, walkers=1021, prec="mixed",
             slater=True, unpaired=2),
        # forces and parameter gradients (the backward direction), FP64 and FP64-equivalent on the tensor cores
        dict(base, name="forces_he16_fp64", kind="forces", atoms=16, recipe=20, walkers=1000),
        dict(base, name="forces_he64_fp64tc", kind="forces", atoms=64, recipe=24, walkers=256, prec="fp64tc"),
        # one stochastic-reconfiguration step: log-derivatives of every lambda entry, then the conjugate gradients
        dict(base, name="sr_he16_fp64", kind="sr", atoms=16, recipe=20, walkers=1024),
        # one lattice-regularised DMC generation: projection and reconfiguration
        dict(base, name="lrdmc_he16_fp64", kind="lrdmc", atoms=16, recipe=20, walkers=1024),
    ]


def draw(rng):
    """One more case: a kind, then sizes over the range that the kind is used in."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = {"kind": rng.choice(["sweep", "sweep", "sweep", "batch", "energy", "forces", "forces", "sr", "lrdmc"])}
    kind = c["kind"]
    c["prec"] = {"sr": "fp64", "lrdmc": rng.choice(["fp64", "fp64tc"]), "batch": rng.choice(["mixed", "fp64"]),
                 "forces": rng.choice(["fp64", "fp64tc"])}.get(kind) or rng.choice(["mixed", "mixed", "fp64", "fp64tc"])
    heavy = c["prec"] == "fp64"  # plain FP64 costs several times the others
    most = {"sweep": 64 if heavy else 160, "batch": 32 if heavy else 64, "energy": 64 if heavy else 128,
            "forces": 32 if heavy else 64, "sr": 16, "lrdmc": 20}[kind]
    c["atoms"] = logint(3, most)
    c["recipe"] = rng.choice([6, 16, 20, 24]) if c["atoms"] <= 64 else 16
    if kind in ("sr", "lrdmc"):
        c["recipe"] = rng.choice([6, 16, 20])
    # walkers: up to about 60 ms of work, and never more than 8192
    per = c["atoms"] * functions(c["recipe"], c["atoms"]) ** 2 * (8 if heavy else 1)
    cap = {"sweep": 4e10, "batch": 1e10, "energy": 4e10, "forces": 1.5e10, "sr": 5e9, "lrdmc": 3e9}[kind] / per
    c["walkers"] = logint(8, max(16, min(8192, cap)))
    c["slater"] = rng.random() < 0.15
    c["band"] = c["atoms"] > 64 or (c["atoms"] > 24 and rng.random() < 0.3)
    c["refresh"] = 16 if kind in ("sweep", "batch") and rng.random() < 0.3 else 0
    c["tune"] = False
    c["unpaired"] = rng.choice([0, 0, 1, 3])
    c["systems"] = rng.randint(2, 8) if kind == "batch" else 1
    return c


def functions(recipe, atoms):
    return atoms * sum(n * k for n, k in zip(RECIPES[recipe], NCOMP))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def sizes(case):
    """(atoms, N_up, N_dn) of each system of the case."""
    out = []
    for s in range(case["systems"]):
        # a batch spreads its systems' sizes evenly down to an eighth of the largest
        f = 1.0 if case["systems"] == 1 else 1.0 - 0.875 * s / (case["systems"] - 1)
        na = max(2, int(round(case["atoms"] * f)))
        if case["recipe"] == 6:  # hydrogen: an electron per atom
            dn = na // 2
            out.append((na, na - dn if not case["unpaired"] else min(na, dn + case["unpaired"]), dn))
        else:                    # helium: a pair per atom, less the unpaired ones' partners
            dn = max(1, na - case["unpaired"] // 2)
            out.append((na, dn + case["unpaired"], dn))
    return out


def make_system(case, index, seed):
    na, nu, nd = sizes(case)[index]
    g = np.random.Generator(np.random.Philox(np.random.SeedSequence([seed, index, 1])))
    hydrogen = case["recipe"] == 6
    side = 3.0 * (na / 4.0) ** (1 / 3) if hydrogen else 10.0 * (na / 16.0) ** (1 / 3)
    sep = 0.5 if hydrogen else 1.5
    R = []
    while len(R) < na:
        p = g.random(3) * side
        if all(((p - q) ** 2).sum() >= sep * sep for q in R):
            R.append(p)
    atom, ls, zeta = [], [], []
    for a in range(na):
        for l, count in enumerate(RECIPES[case["recipe"]]):
            for z in sorted(np.exp(g.uniform(math.log(0.1), math.log(10.0), size=count)), reverse=True):
                atom.append(a)
                ls.append(l)
                zeta.append(z)
    L = sum(NCOMP[l] for l in ls)
    radial = np.zeros(len(ls), np.int32)
    if case["slater"]:
        radial = (g.random(len(ls)) < 0.3).astype(np.int32)
        zeta = np.where(radial == 1, 0.5 + g.random(len(ls)), zeta)
    lam = g.standard_normal((L, L)) * 0.1
    lam = np.triu(lam) + np.triu(lam, 1).T
    lam[np.diag_indices(L)] += 1.0
    if case["band"]:  # about a tenth of the entries, stored dense
        w = max(1, L // 20)
        lam = np.triu(np.tril(lam, w), -w)
    unpaired = g.normal(0.0, 0.5, size=(nu - nd, L)) if nu > nd else None
    sysm = SimpleNamespace(
        R=np.array(R), Z=np.full(na, 1.0 if hydrogen else 2.0), shell_atom=np.array(atom, np.int32),
        shell_l=np.array(ls, np.int32), shell_radial=radial, shell_zeta=np.array(zeta, np.float64), lam=lam, L=L,
        n_up=nu, n_dn=nd, unpaired=unpaired, b_ea=1.0, b_para=1.0, b_anti=1.0, use_j1=not hydrogen, use_j2=True,
        j2_spin_independent=hydrogen, delta=1.6 if hydrogen else 1.5, j3=None)
    centres = np.array([R[i % na] for i in range(nu)] + [R[(j + na // 2) % na] for j in range(nd)])
    x = centres[None] + g.uniform(-1.0, 1.0, size=(case["walkers"], nu + nd, 3))
    return sysm, x


def prepare(case, seed):
    """Handles, walker states evaluated at the starting positions, and the positions."""
    members, pos, start = [], [], []
    for s in range(case["systems"]):
        sysm, x = make_system(case, s, seed)
        g = pg.JAGP(sysm, case["walkers"], precision=pg.JAGP_PREC_MIXED if case["prec"] == "mixed" else pg.JAGP_PREC_FP64,
                    seed=seed, refresh_moves=case["refresh"], fp64_tc=case["prec"] == "fp64tc")
        r = g.positions(x)
        if case["tune"]:
            g.autotune()
        g.eval(r)
        members.append(g)
        pos.append(r)
    st = {"case": case, "g": members, "r": pos, "sweep": 0}
    if case["kind"] == "batch":
        st["batch"] = pg.Batch(members, pos)
    if case["kind"] == "sr":
        W, P = case["walkers"], members[0].sys.L ** 2 + 3
        st["O"] = torch.empty((W, P), dtype=torch.float64, device="cuda")
        st["eL"] = members[0].local_energy(pos[0])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    kind, g, r = state["case"]["kind"], state["g"][0], state["r"][0]
    t = state["sweep"]
    state["sweep"] += 1
    if kind == "sweep":
        eL, acc = g.sweep(r, 1, sweep0=t, acc=True)
        return {"r": r, "eL": eL[0], "acc": acc[0]}
    if kind == "batch":
        b = state["batch"]
        b.sweep(1, sweep0=t)
        return {"r": b.r, "eL": b.eL}
    if kind == "energy":
        logabs, sign = g.eval(r)
        eL, parts = g.local_energy(r, parts=True)
        return {"logabs": logabs, "sign": sign, "eL": eL, "parts": parts}
    if kind == "forces":
        eL = g.local_energy(r)
        sL, sE, mean = pg.jagp_force_seeds(eL)
        out = g.grad(r, seed_logpsi=sL, seed_eL=sE)
        pg.jagp_space_warp(g.h, r, r.shape[0], out["r"], out["R_walker"], sL, out["R"])
        return dict(out, mean=mean)
    if kind == "sr":
        g.logpsi_derivs(r, state["O"])
        f, step, _, _ = pg.jagp_sr_step(state["O"], state["eL"], eps=1e-2, max_iter=SR_ITERS, tol=1e-12)
        return {"O": state["O"], "f": f, "step": step}
    out = g.lrdmc(r, 1, a=LRDMC_A, tau=LRDMC_TAU, gen0=t)
    return {"r": r, **{k: out[k] for k in ("wbar", "ebar", "eL", "weight", "hops", "parent")}}


def work(case):
    """Operations and bytes of one pass that no form of the method avoids: inputs, results and lambda once; the lambda
    rows of accepted moves (about half), the rows of G~ per proposal, G~ and the kinetic vectors."""
    flops = nbytes = 0.0
    W, kind = case["walkers"], case["kind"]
    for s, (na, nu, nd) in enumerate(sizes(case)):
        N, L = nu + nd, functions(case["recipe"], na)
        density = 0.1 if case["band"] else 1.0
        row, geminal, mvec, basis = 2.0 * L * L * density, 2.0 * nu * nu * L, 2.0 * N * nu * L, 30.0 * N * L
        energy = mvec + basis + 60.0 * N * (N + na)
        nbytes += 8.0 * (L * L * density + W * (2 * 3 * N + 2))
        if kind in ("sweep", "batch"):
            flops += W * (0.5 * N * row + 2.0 * N * nu * L + geminal + basis + energy + 6.0 * 0.5 * N * nu * nu)
        elif kind == "energy":
            flops += W * (N * row + geminal + basis + energy)
        elif kind == "forces":
            flops += W * (2 * energy + (2 * N) * row / density + 6 * mvec)
            nbytes += 8.0 * L * L
        elif kind == "sr":
            flops += W * (2.0 * nu * L * L + 2.0 * nu * nd * L) + SR_ITERS * 4.0 * W * L * L
            nbytes += 8.0 * W * L * L * (1 + SR_ITERS)
        else:
            hops = 12.0  # a generation's hops per walker at this tau, about
            flops += W * (N * row + geminal + energy + hops * (row + geminal + energy + 12.0 * N * L))
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the method in float64 torch (one system), for `exact`
# ---------------------------------------------------------------------------
class Model:
    def __init__(self, sysm, seed):
        self.s, self.seed = sysm, seed
        t = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda")  # noqa: E731
        self.R, self.Z, self.lam = t(sysm.R), t(sysm.Z), t(sysm.lam)
        self.unp = None if sysm.unpaired is None else t(sysm.unpaired)
        self.c = (2.0 * self.Z) ** 0.25
        self.b = torch.tensor([sysm.b_ea, sysm.b_para, sysm.b_anti], dtype=torch.float64, device="cuda")
        off = np.concatenate([[0], np.cumsum([NCOMP[l] for l in sysm.shell_l])])
        order, self.groups = [], []
        for rad in (0, 1):
            for l in (0, 1, 2):
                k = np.nonzero((sysm.shell_l == l) & (sysm.shell_radial == rad))[0]
                if len(k):
                    self.groups.append((l, rad, torch.as_tensor(sysm.shell_atom[k].astype(np.int64), device="cuda"),
                                        t(sysm.shell_zeta[k])))
                    order.append((off[k][:, None] + np.arange(NCOMP[l])).reshape(-1))
        self.perm = torch.as_tensor(np.argsort(np.concatenate(order)), device="cuda")
        nu, N = sysm.n_up, sysm.n_up + sysm.n_dn
        up = torch.arange(N, device="cuda") < nu
        self.same = (up[:, None] == up[None]) & (not sysm.j2_spin_independent)
        self.kk = torch.where(self.same, 4.0, 2.0).double()
        iu = torch.triu_indices(self.Z.numel(), self.Z.numel(), 1, device="cuda")
        self.iu = iu

    def bb(self, b):
        return torch.where(self.same, b[1], b[2])

    def orbitals(self, x, R=None, derivs=False):
        """Values [..., L] at points x [..., 3]; with derivs also gradients [..., L, 3] and Laplacians."""
        R = self.R if R is None else R
        v, g, lp = [], [], []
        for l, rad, atom, zeta in self.groups:
            d = x[..., None, :] - R[atom]
            dx, dy, dz = d.unbind(-1)
            r2 = (d * d).sum(-1)
            if rad:
                r = r2.sqrt()
                e = torch.exp(-zeta * r)
                q = -zeta / r * e
                le = (zeta * zeta - 2.0 * zeta / r) * e
            else:
                e = torch.exp(-zeta * r2)
                q = -2.0 * zeta * e
                le = (4.0 * zeta * zeta * r2 - 6.0 * zeta) * e
            one, zero = torch.ones_like(dx), torch.zeros_like(dx)
            if l == 0:
                P, dP = [one], [(zero, zero, zero)]
            elif l == 1:
                P, dP = [dx, dy, dz], [(one, zero, zero), (zero, one, zero), (zero, zero, one)]
            else:
                P = [dx * dy, dy * dz, dz * dx, dx * dx - dy * dy, 3.0 * dz * dz - r2]
                dP = [(dy, dx, zero), (zero, dz, dy), (dz, zero, dx), (2 * dx, -2 * dy, zero), (-2 * dx, -2 * dy, 4 * dz)]
            v.append(torch.stack([p * e for p in P], -1).flatten(-2))
            if derivs:
                # harmonic polynomials of degree l: grad P . d = l P, lap P = 0
                g.append(torch.stack([torch.stack([gp[k] * e + p * q * (dx, dy, dz)[k] for k in range(3)], -1)
                                      for p, gp in zip(P, dP)], -2).flatten(-3, -2))
                lp.append(torch.stack([2.0 * l * p * q + p * le for p in P], -1).flatten(-2))
        cat = lambda a, dim: torch.cat(a, dim).index_select(dim, self.perm)  # noqa: E731
        return (cat(v, -1), cat(g, -2), cat(lp, -1)) if derivs else cat(v, -1)

    def bt_rows(self, phi_dn, lam=None):
        bt = phi_dn @ (self.lam if lam is None else lam).T
        return bt if self.unp is None else torch.cat([bt, self.unp.expand(bt.shape[0], -1, -1)], 1)

    def jastrow(self, x, R=None, b=None):
        """J, gradients [W, N, 3] and Laplacians [W, N]."""
        R, b = (self.R if R is None else R), (self.b if b is None else b)
        J = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
        g, lp = torch.zeros_like(x), torch.zeros_like(x[..., 0])
        if self.s.use_j1:
            d = x[:, :, None] - R
            r = d.norm(dim=-1)
            c = self.c
            e = torch.exp(-b[0] * c * r)
            f1, f2 = -0.5 * c ** 4 * e, 0.5 * c ** 5 * b[0] * e
            J = J - (c ** 3 * (1.0 - e) / (2.0 * b[0])).sum((1, 2))
            g = g + (f1 / r)[..., None].mul(d).sum(2)
            lp = lp + (f2 + 2.0 * f1 / r).sum(2)
        if self.s.use_j2:
            N = x.shape[1]
            eye = torch.eye(N, dtype=torch.bool, device="cuda")
            d = x[:, :, None] - x[:, None]
            r = torch.where(eye, 1.0, (d * d).sum(-1)).sqrt()
            bb = self.bb(b)
            q = 1.0 + bb * r
            off = (~eye).double()
            J = J + 0.5 * (off * r / (self.kk * q)).sum((1, 2))
            v1 = off / (self.kk * q * q)
            g = g + (v1 / r)[..., None].mul(d).sum(2)
            lp = lp + (-2.0 * bb * v1 / q + 2.0 * v1 / r).sum(2)
        return J, g, lp

    def coulomb(self, x, R=None):
        R = self.R if R is None else R
        N = x.shape[1]
        vei = -(self.Z / (x[:, :, None] - R).norm(dim=-1)).sum((1, 2))
        i, j = torch.triu_indices(N, N, 1, device="cuda")
        vee = (1.0 / (x[:, i] - x[:, j]).norm(dim=-1)).sum(1)
        a, c = self.iu
        vii = (self.Z[a] * self.Z[c] / (R[a] - R[c]).norm(dim=-1)).sum()
        return vee, vei, vii

    def evaluate(self, x, R=None, lam=None, b=None):
        """log|Psi|, sign, e_L, (kinetic, V_ee, V_ei, V_ii), the kinetic vectors M."""
        nu, nd = self.s.n_up, self.s.n_dn
        L = self.lam if lam is None else lam
        v, g, lp = self.orbitals(x, R, derivs=True)
        bt = self.bt_rows(v[:, nu:], L)
        a = v[:, :nu] @ L
        G = v[:, :nu] @ bt.transpose(1, 2)
        sign, logdet = torch.linalg.slogdet(G)
        Gi = torch.linalg.inv(G)
        M = torch.cat([Gi.transpose(1, 2) @ bt, Gi[:, :nd] @ a], 1)
        gD, lD = (g * M[..., None]).sum(2), (lp * M).sum(2)
        J, gJ, lJ = self.jastrow(x, R, b)
        kin = -0.5 * (lD + lJ + 2.0 * (gD * gJ).sum(-1) + (gJ * gJ).sum(-1)).sum(1)
        vee, vei, vii = self.coulomb(x, R)
        return logdet + J, sign, kin + vee + vei + vii, (kin, vee, vei, vii), M

    def chunked(self, x, f):
        step = max(1, int(4e7 / (x.shape[1] * self.s.L)))
        out = [f(x[k:k + step]) for k in range(0, x.shape[0], step)]
        return [torch.cat(o) for o in zip(*out)]

    def energies(self, x):
        def f(y):
            la, sg, e, (k, ee, ei, ii), M = self.evaluate(y)
            return la, sg, e, torch.stack([k, ee, ei, ii.expand_as(k)], 1)
        return self.chunked(x, f)

    def draws(self, W, sweep, electrons, last=1):
        """Philox4x32-10 words [4][W][len(electrons)] of counters (walker, sweep, electron, last)."""
        c = [np.broadcast_to(np.arange(W, dtype=np.uint64)[:, None], (W, len(electrons))),
             np.full((W, len(electrons)), sweep, np.uint64),
             np.broadcast_to(np.asarray(electrons, np.uint64)[None], (W, len(electrons))),
             np.full((W, len(electrons)), last, np.uint64)]
        lo = np.uint64(0xFFFFFFFF)
        k0, k1 = self.seed & 0xFFFFFFFF, self.seed >> 32
        for _ in range(10):
            p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
            c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & lo, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & lo]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        return torch.as_tensor(np.stack(c).astype(np.float64), device="cuda")

    def sweep(self, x, t):
        """One Metropolis sweep (up electrons, then down); returns positions and the accepted moves."""
        nu, nd = self.s.n_up, self.s.n_dn
        x, W = x.clone(), x.shape[0]
        accepted = torch.zeros((), dtype=torch.float64, device="cuda")
        phi_up = self.chunked(x, lambda y: (self.orbitals(y[:, :nu]),))[0]
        bt = self.chunked(x, lambda y: (self.bt_rows(self.orbitals(y[:, nu:])),))[0]
        for up in (True, False):
            n, e0 = (nu, 0) if up else (nd, nu)
            if n == 0:
                continue
            u = self.draws(W, t, list(range(e0, e0 + n)))
            prop = x[:, e0:e0 + n] + self.s.delta * ((u[:3] + 0.5) * 2.0 ** -31 - 1.0).permute(1, 2, 0)
            table = bt if up else self.chunked(phi_up, lambda y: (y @ self.lam,))[0]
            phi_new = self.chunked(prop, lambda y: (self.orbitals(y),))[0]
            rows = phi_new @ table.transpose(1, 2)            # proposed rows (up) or columns (down)
            Gi = torch.linalg.inv(phi_up @ bt.transpose(1, 2))
            if not up:
                Gi = Gi.transpose(1, 2).contiguous()            # a column move is a row move of the transpose
            w = torch.arange(W, device="cuda")
            for m in range(n):
                ratio = (rows[:, m] * Gi[:, :, m]).sum(1)
                dJ = self.delta_j(x, e0 + m, prop[:, m])
                p = ratio ** 2 * torch.exp(2.0 * dJ)
                ok = (u[3, :, m] * 2.0 ** -32 < p) & (ratio != 0)
                col = Gi[:, :, m].clone()
                vec = torch.einsum("wj,wjk->wk", rows[:, m], Gi)
                vec[:, m] -= 1.0
                scale = torch.where(ok, 1.0 / ratio, torch.zeros_like(ratio))
                Gi -= (col * scale[:, None])[:, :, None] * vec[:, None]
                x[w[ok], e0 + m] = prop[ok, m]
                accepted += ok.sum()
            if up:
                phi_up = self.chunked(x, lambda y: (self.orbitals(y[:, :nu]),))[0]
        return x, accepted

    def delta_j(self, x, e, new):
        out = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
        if self.s.use_j1:
            f = lambda y: (self.c ** 3 * (1.0 - torch.exp(-self.b[0] * self.c * (y[:, None] - self.R).norm(dim=-1)))  # noqa: E731
                           / (2.0 * self.b[0])).sum(1)
            out += f(x[:, e]) - f(new)
        if self.s.use_j2:
            k, b = self.kk[e].clone(), self.bb(self.b)[e]
            k[e] = math.inf
            f = lambda y: ((y[:, None] - x).norm(dim=-1) / (k * (1.0 + b * (y[:, None] - x).norm(dim=-1)))).sum(1)  # noqa: E731
            out += f(new) - f(x[:, e])
        return out

    def forces(self, x):
        W, na = x.shape[0], self.Z.numel()
        e = self.energies(x)[2]
        E = e.mean()
        sL, sE = 2.0 * (e - E) / W, torch.full_like(e, 1.0 / W)
        lam, b = self.lam.clone().requires_grad_(), self.b.clone().requires_grad_()
        eL, dx, dRw, dlam, db = [], [], [], 0.0, 0.0
        step = max(1, int(4e6 / (x.shape[1] * self.s.L)))
        for k in range(0, W, step):
            y = x[k:k + step].clone().requires_grad_()
            # a copy of R per walker gives the per-walker derivatives
            w = y.shape[0]
            Rw = self.R.expand(w, na, 3).clone().requires_grad_()
            la, _, el, _, _ = self._evaluate_R(y, Rw, lam, b)
            lj = self.jastrow_R(y.detach(), Rw.detach(), b)
            s = slice(k, k + step)
            gy, gR, gl = torch.autograd.grad((sL[s] * la + sE[s] * el).sum(), (y, Rw, lam))
            gb, = torch.autograd.grad((sL[s] * lj).sum(), (b,))
            eL.append(el.detach())
            dx.append(gy)
            dRw.append(gR)
            dlam, db = dlam + gl, db + gb
        dx, dRw = torch.cat(dx), torch.cat(dRw)
        # space warp: omega_a = kappa_a / sum kappa, kappa = 1 / r^4
        d = x[:, :, None] - self.R
        r2 = (d * d).sum(-1)
        kap = 1.0 / (r2 * r2)
        S = kap.sum(2, keepdim=True)
        om = kap / S
        gk = (-4.0 * kap / r2)[..., None] * d
        gom = gk / S[..., None] - (kap / (S * S))[..., None] * gk.sum(2, keepdim=True)
        dRw = dRw + torch.einsum("wia,wiq->waq", om, dx) + 0.5 * sL[:, None, None] * gom.sum(1)
        # d J / d b of parameters that the wave function does not use is zero
        return {"eL": torch.cat(eL), "lam": dlam, "jas": db, "R": dRw.sum(0), "R_walker": dRw, "r": dx,
                "mean": torch.stack([E, torch.ones_like(E)])}

    def _evaluate_R(self, y, Rw, lam, b):
        """evaluate() with a copy of the nuclear positions per walker: the walker axis is carried by broadcasting."""
        return self.evaluate_with(y, Rw, lam, b)

    def evaluate_with(self, y, Rw, lam, b):
        nu, nd = self.s.n_up, self.s.n_dn
        v, g, lp = self.orbitals_R(y, Rw)
        bt = self.bt_rows(v[:, nu:], lam)
        a = v[:, :nu] @ lam
        G = v[:, :nu] @ bt.transpose(1, 2)
        sign, logdet = torch.linalg.slogdet(G)
        Gi = torch.linalg.inv(G)
        M = torch.cat([Gi.transpose(1, 2) @ bt, Gi[:, :nd] @ a], 1)
        gD, lD = (g * M[..., None]).sum(2), (lp * M).sum(2)
        J, gJ, lJ = self.jastrow(y, Rw[:, None], b.detach())
        kin = -0.5 * (lD + lJ + 2.0 * (gD * gJ).sum(-1) + (gJ * gJ).sum(-1)).sum(1)
        N = y.shape[1]
        vei = -(self.Z / (y[:, :, None] - Rw[:, None]).norm(dim=-1)).sum((1, 2))
        i, j = torch.triu_indices(N, N, 1, device="cuda")
        vee = (1.0 / (y[:, i] - y[:, j]).norm(dim=-1)).sum(1)
        p, q = self.iu
        vii = (self.Z[p] * self.Z[q] / (Rw[:, p] - Rw[:, q]).norm(dim=-1)).sum(1)
        return logdet + J, sign, kin + vee + vei + vii, None, M

    def orbitals_R(self, y, Rw):
        class PerWalker:  # indexed by atom like R, with the walker axis in front
            def __getitem__(_, atom):
                return Rw[:, None, atom]
        return self.orbitals(y, PerWalker(), derivs=True)

    def jastrow_R(self, y, Rw, b):
        return self.jastrow(y, Rw[:, None], b)[0]

    def log_derivatives(self, x):
        nu, nd = self.s.n_up, self.s.n_dn

        def f(y):
            v = self.orbitals(y)
            bt = self.bt_rows(v[:, nu:])
            Gi = torch.linalg.inv(v[:, :nu] @ bt.transpose(1, 2))
            Y = Gi[:, :nd].transpose(1, 2) @ v[:, nu:]
            O = v[:, :nu].transpose(1, 2) @ Y
            s = self.s
            j = torch.zeros((y.shape[0], 3), dtype=torch.float64, device="cuda")
            if s.use_j1:
                sc, b = self.c * (y[:, :, None] - self.R).norm(dim=-1), self.b[0]
                e = torch.exp(-b * sc)
                j[:, 0] = -(self.c ** 3 * (sc * e / (2 * b) - (1 - e) / (2 * b * b))).sum((1, 2))
            if s.use_j2:
                r = (y[:, :, None] - y[:, None]).norm(dim=-1)
                d = -0.5 * r * r / (self.kk * (1.0 + self.bb(self.b) * r) ** 2)
                j[:, 1] = (d * self.same).sum((1, 2))
                j[:, 2] = (d * ~self.same).sum((1, 2))
            return (torch.cat([O.flatten(1), j], 1),)
        return self.chunked(x, f)[0]

    def lrdmc(self, x, a, tau, gen):
        """One continuous-time projection and the reconfiguration."""
        x, (W, N) = x.clone(), x.shape[:2]
        s = self.s
        left, lw = torch.full((W,), tau, dtype=torch.float64, device="cuda"), torch.zeros(W, dtype=torch.float64, device="cuda")
        hops, e = torch.zeros(W, dtype=torch.int32, device="cuda"), torch.empty(W, dtype=torch.float64, device="cuda")
        M = torch.empty((W, N, s.L), dtype=torch.float64, device="cuda")
        live = torch.arange(W, device="cuda")
        step = torch.zeros((6, 3), dtype=torch.float64, device="cuda")
        for d in range(3):
            step[2 * d, d], step[2 * d + 1, d] = a, -a
        while live.numel():
            parts = self.chunked(x[live], lambda y: self.evaluate(y)[2:5:2])
            e[live], M[live] = parts[0], parts[1]
            rho = torch.empty((live.numel(), N, 6), dtype=torch.float64, device="cuda")
            for i in range(N):
                new = x[live, i][:, None] + step
                det = torch.einsum("wkl,wl->wk", self.orbitals(new), M[live, i])
                dj = torch.stack([self.delta_j(x[live], i, new[:, k]) for k in range(6)], 1)
                rho[:, i] = det * torch.exp(dj)
            rate = torch.where(rho > 0, rho, torch.zeros_like(rho)).flatten(1) / (2.0 * a * a)
            run = rate.cumsum(1)
            G = run[:, -1]
            u = torch.as_tensor(np.stack([self.hop_draw(int(w), gen, int(h)) for w, h in zip(live.tolist(), hops[live].tolist())]),
                                device="cuda")
            wait = -torch.log(1.0 - u[:, 0]) / G
            stop = wait >= left[live]
            dt = torch.where(stop, left[live], wait)
            lw[live] -= dt * e[live]
            left[live] -= dt
            k = (run > (u[:, 1] * G)[:, None]).int().argmax(1)
            move = live[~stop]
            km = k[~stop]
            x[move, km // 6] += step[km % 6]
            hops[move] += 1
            live = move
        w = torch.exp(lw)
        z = (float(self.draws(1, gen, [0], last=3)[0, 0, 0]) + 0.5) * 2.0 ** -32
        wsum = w.cumsum(0)
        thr = (torch.arange(W, dtype=torch.float64, device="cuda") + z) * wsum[-1] / W
        parent = torch.searchsorted(wsum, thr, right=True).clamp(max=W - 1)
        return {"r": x[parent], "wbar": (wsum[-1] / W)[None], "ebar": ((w * e).sum() / wsum[-1])[None], "eL": e[None],
                "weight": w[None], "hops": hops[None], "parent": parent.int()[None]}

    def hop_draw(self, walker, gen, hop):
        lo = 0xFFFFFFFF
        c, k0, k1 = [walker, gen, hop, 2], self.seed & lo, self.seed >> 32
        for _ in range(10):
            p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
            c = [(p1 >> 32) ^ c[1] ^ k0, p1 & lo, (p0 >> 32) ^ c[3] ^ k1, p0 & lo]
            k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
        return np.array([(c[0] + 0.5) * 2.0 ** -32, (c[1] + 0.5) * 2.0 ** -32])


def exact(case, seed):
    models = []
    for s in range(case["systems"]):
        sysm, x = make_system(case, s, seed)
        models.append((Model(sysm, seed), torch.as_tensor(x, device="cuda")))
    m, x = models[0]
    kind = case["kind"]
    with torch.set_grad_enabled(kind == "forces"):
        if kind in ("sweep", "batch"):
            # a chain's acceptances follow the FP32 ratios in mixed precision: its positions and energies have this
            # value up to moves whose draw falls within that rounding
            out = {"r": [], "eL": []}
            for mm, xx in models:
                y, n = mm.sweep(xx, 0)
                e = mm.energies(y)[2]
                out["r"].append(y)
                out["eL"].append(e)
            if kind == "batch":
                return out
            return {"r": out["r"][0], "eL": out["eL"][0], "acc": None}
        if kind == "energy":
            la, sg, e, parts = m.energies(x)
            return {"logabs": la, "sign": sg, "eL": e, "parts": parts}
        if kind == "forces":
            return m.forces(x)
        if kind == "sr":
            O = m.log_derivatives(x)
            e = m.energies(x)[2]
            f = -2.0 / x.shape[0] * ((e - e.mean()) @ (O - O.mean(0)))
            return {"O": O, "f": f, "step": None}
        return m.lrdmc(x, LRDMC_A, LRDMC_TAU, 0)
