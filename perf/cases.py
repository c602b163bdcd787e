"""What the engine is measured on: calls that programs built on it make, over the sizes they make them at.

Kinds of case
  md         trajectories from given states: mw_set_state_dev (isobaric: the restore of a checkpoint), mw_step with
             its thermo record, mw_get_state_dev (an external driver's single step, sampling segments, replica
             batches, isobaric scans, the slab)
  frames     single-point energies, forces and virials of unrelated snapshots, one after another
  fit        force matching: forces and their adjoint at two parameter sets (an iterate and a trial step) of a
             batch of frames, through torch autograd
  structure  g(r) and angle histograms of a frame

Inputs are seeded synthetic boxes.  Liquids start on a jittered grid and are settled for a few tens of steps by the
plain FP64 dynamics below, so that the neighbour counts, forces and speeds are a liquid's; the 10^6-atom cases start
from jittered lattices (settling them here would take longer than measuring them).  The FP64 reference (exact) is
plain torch: a half pair list, the total energy in closed form, its derivatives by autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0809_2811_gb300 import mw, torch_ops

# ------------------------------------------------------------------ the cases


def listed():
    return [
        # one NVE step of the smallest box, state in and out: a driver that integrates something else around it
        {"name": "md_512_step1", "kind": "md", "boxes": 1, "n": 512, "ensemble": "nve", "steps": 1},
        # the same box, a segment between records
        {"name": "md_512_nve_50", "kind": "md", "boxes": 1, "n": 512, "ensemble": "nve", "steps": 50},
        # the usual size of a property run, Nose-Hoover
        {"name": "md_4096_nh_50", "kind": "md", "boxes": 1, "n": 4096, "ensemble": "nh", "steps": 50},
        # isobaric density scan: eight boxes, each with its own barostat, a segment from a checkpoint
        {"name": "npt_8x4096_40", "kind": "md", "boxes": 8, "n": 4096, "ensemble": "npt", "steps": 40},
        # ice and liquid side by side as two boxes of one batch, with the wider skin that long runs use
        {"name": "md_2x32768_nh_25", "kind": "md", "boxes": 2, "n": 32768, "ensemble": "nh", "steps": 25, "ice": True,
         "skin": 2.6},
        # cooling / density scan: 256 boxes of uneven size, density and temperature
        {"name": "md_batch256_nh_20", "kind": "md", "boxes": 256, "n": 8000, "n_min": 216, "ensemble": "nh",
         "steps": 20},
        # ice slab in contact with liquid, 2^20 atoms, graph engine with the skin that suits it
        {"name": "md_slab_1m_nh_16", "kind": "md", "system": "slab", "boxes": 1, "n": 1048576, "ensemble": "nh",
         "steps": 16, "skin": 2.0, "engine": "graph"},
        # water with a tenth of solute particles (two species)
        {"name": "solute_32768_nh_20", "kind": "md", "boxes": 1, "n": 32768, "ensemble": "nh", "steps": 20,
         "solute": 0.1},
        # energies and forces of snapshots: a small box, and a large one
        {"name": "frames_512", "kind": "frames", "boxes": 1, "n": 512, "frames": 4},
        {"name": "frames_32768", "kind": "frames", "boxes": 1, "n": 32768, "frames": 4},
        # a force-matching iteration over a training set
        {"name": "fit_64x4096", "kind": "fit", "boxes": 64, "n": 4096},
        # structure of an ice and a liquid frame
        {"name": "structure_2x32768", "kind": "structure", "boxes": 2, "n": 32768, "ice": True, "skin": 1.5},
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["md", "md", "md", "batch", "npt", "solute", "frames", "fit", "structure"])
    if kind == "md":
        n = logint(300, 200000)
        return {"kind": "md", "boxes": 1, "n": n, "ensemble": rng.choice(["nve", "nh"]),
                "steps": logint(1, 50 if n < 20000 else 20), "skin": rng.choice([1.0, 1.0, 1.6, 2.2])}
    if kind == "batch":
        n = logint(400, 8000)
        return {"kind": "md", "boxes": logint(2, 100), "n": n, "n_min": max(216, n // 10), "ensemble": "nh",
                "steps": logint(5, 25)}
    if kind == "npt":
        return {"kind": "md", "boxes": logint(1, 12), "n": logint(500, 6000), "ensemble": "npt", "steps": logint(10, 40)}
    if kind == "solute":
        return {"kind": "md", "boxes": 1, "n": logint(1500, 60000), "ensemble": "nh", "steps": logint(2, 25),
                "solute": round(rng.uniform(0.03, 0.3), 3)}
    if kind == "frames":
        return {"kind": "frames", "boxes": 1, "n": logint(300, 100000), "frames": rng.randint(2, 4)}
    if kind == "fit":
        return {"kind": "fit", "boxes": logint(1, 50), "n": logint(300, 5000)}
    return {"kind": "structure", "boxes": logint(1, 4), "n": logint(1000, 30000), "skin": 1.5}


# ------------------------------------------------------------------ the model in FP64 (plain torch)

KB, FCONV, ATM, MASS = 0.0019872042586408316, 4.184e-4, 68568.4158, 18.015
VMOL = MASS / 6.02214076e23 * 1e24  # A^3 per molecule at 1 g/cm^3
LAM, EPS, SIG, A_, GAM, AA, BB, C0 = 23.15, 6.189, 2.3925, 1.8, 1.2, 7.049556277, 0.6022245584, -1.0 / 3.0
F64 = torch.float64


class Model:
    """Boxes, species constants and the pair list of a configuration."""

    def __init__(self, n, L, types=None, theta=None, pad=0.6):
        self.n = torch.as_tensor(n, device="cuda")
        self.L = torch.as_tensor(L, dtype=F64, device="cuda").reshape(len(n), 3)
        self.bid = torch.repeat_interleave(torch.arange(len(n), device="cuda"), self.n)
        self.types = types
        lam, eps, sig = (LAM, EPS, SIG) if theta is None else theta
        if types is None:  # 1 x 1 tables
            self.eps, self.sig, self.lam = (torch.as_tensor(v, dtype=F64, device="cuda") for v in (eps, sig, lam))
            self.rc = A_ * float(sig)
        else:  # water, solute: two-body terms only for the solute
            t = solute_table()
            pair = torch.tensor(np.array([[t[a, b, b] for b in range(2)] for a in range(2)]), dtype=F64, device="cuda")
            self.lam, self.eps, self.sig = pair[..., 0], pair[..., 1], pair[..., 2]
            self.rc = A_ * float(self.sig.max())
        self.pad, self.x_list = pad, None

    def pairs(self, x):
        """Half list (i, j) of the pairs within rc + pad, kept while no atom has moved pad / 2."""
        if self.x_list is not None:
            d = x - self.x_list
            lb = self.L[self.bid]
            if float((d - lb * torch.round(d / lb)).square().sum(1).max()) < (0.5 * self.pad) ** 2 * 0.98:
                return self.ij
        r = self.rc + self.pad
        nc = torch.floor(self.L / r).long()
        assert int(nc.min()) >= 3, "boxes of at least three cells an edge"
        ncell = nc.prod(1)
        off = torch.cumsum(ncell, 0) - ncell
        s = x / self.L[self.bid]
        s = s - torch.floor(s)
        ncb = nc[self.bid]
        c = torch.minimum((s * ncb).long(), ncb - 1)

        def cell(q):
            return off[self.bid] + q[:, 0] + ncb[:, 0] * (q[:, 1] + ncb[:, 1] * q[:, 2])

        me = cell(c)
        order = torch.argsort(me, stable=True)
        cnt = torch.bincount(me, minlength=int(ncell.sum()))
        start = torch.cumsum(cnt, 0) - cnt
        idx = torch.arange(len(x), device="cuda")
        ii, jj = [], []
        for o in range(13, 27):  # the cell itself and 13 of its 26 neighbours
            shift = torch.tensor([o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1], device="cuda")
            there = cell((c + shift) % ncb)
            k = cnt[there]
            i = torch.repeat_interleave(idx, k)
            first = torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
            j = order[start[there][i] + torch.arange(len(i), device="cuda") - first]
            if o == 13:
                i, j = i[i < j], j[i < j]
            near = self.vec(x, i, j).square().sum(1) < r * r
            ii.append(i[near])
            jj.append(j[near])
        self.x_list, self.ij = x.clone(), (torch.cat(ii), torch.cat(jj))
        return self.ij

    def vec(self, x, i, j):
        lb = self.L[self.bid[i]]
        d = x[j] - x[i]
        return d - lb * torch.round(d / lb)

    def terms(self, d, i, j):
        """E2 per pair and E3 per atom.  With e = sqrt(lam eps) exp(gam sig / (r - a sig)), u = d / r and the sums
        S = sum e, s = sum e u, M = sum e u u^T over an atom's legs, its angle sum over leg pairs is
        (|M|^2 - 2 c0 |s|^2 + c0^2 S^2 - (1 - c0)^2 sum e^2) / 2."""
        eps, sig, lam = self.eps, self.sig, self.lam
        if self.types is not None:
            ti, tj = self.types[i], self.types[j]
            eps, sig, lam = eps[ti, tj], sig[ti, tj], lam[ti, tj]
        r = d.square().sum(1).sqrt()
        t = 1.0 / (r - A_ * sig)
        e2 = AA * eps * (BB * (sig / r) ** 4 - 1.0) * torch.exp(sig * t)
        e = torch.exp(GAM * sig * t) * (torch.sqrt(lam * eps) if self.types is None else torch.sqrt(lam.detach() * eps))
        u = d / r[:, None]
        eu = e[:, None] * u
        uu = (eu[:, :, None] * u[:, None, :]).reshape(-1, 9)
        zero = torch.zeros(len(self.bid), 14, dtype=F64, device="cuda")
        both = torch.cat([uu, (e * e)[:, None], e[:, None]], 1)
        m = zero.index_add(0, i, torch.cat([both, eu], 1)).index_add(0, j, torch.cat([both, -eu], 1))
        q = m[:, :9].square().sum(1) - 2 * C0 * m[:, 11:].square().sum(1) + (C0 * m[:, 10]) ** 2
        return e2, 0.5 * (q - (1 - C0) ** 2 * m[:, 9])

    def legs(self, x):
        i, j = self.pairs(x)
        r2 = self.vec(x, i, j).square().sum(1)
        rc = self.rc if self.types is None else A_ * self.sig[self.types[i], self.types[j]]
        near = r2 < rc * rc * (1 - 1e-13)
        return i[near], j[near]

    def evaluate(self, x):
        """Forces, (E, E2, E3) and the virial of every box."""
        i, j = self.legs(x)
        d = self.vec(x, i, j).requires_grad_()
        e2, e3 = self.terms(d, i, j)
        g, = torch.autograd.grad(e2.sum() + e3.sum(), d)
        d = d.detach()
        f = torch.zeros_like(x).index_add_(0, i, g).index_add_(0, j, -g)
        zb = torch.zeros(len(self.n), dtype=F64, device="cuda")
        s2 = zb.index_add(0, self.bid[i], e2.detach())
        s3 = zb.index_add(0, self.bid, e3.detach())
        w = torch.zeros(len(self.n), 6, dtype=F64, device="cuda")
        w.index_add_(0, self.bid[i], -torch.stack([d[:, a] * g[:, b] for a, b in
                                                    ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1))
        return f, torch.stack([s2 + s3, s2, s3], 1), w

    def per_atom(self, v):
        return v[self.bid][:, None]

    def kinetic(self, v):
        k = 0.5 * MASS / FCONV * v.square().sum(1)
        return torch.zeros(len(self.n), dtype=F64, device="cuda").index_add_(0, self.bid, k)


def dynamics(m, x, v, steps, ensemble, T, dt=10.0, tau=1000.0, p=0.0, tau_p=2500.0):
    """Velocity Verlet in FP64: "nve", "nh" (one Nose-Hoover thermostat a box, half steps around the Verlet step),
    "npt" (with the isotropic barostat inside those half steps) or "scale" (speeds scaled to T after each step)."""
    ndf = 3.0 * m.n.to(F64) - 3.0
    T = torch.as_tensor(T, dtype=F64, device="cuda").expand(len(m.n))
    kT = KB * T
    Q, W = ndf * kT * tau * tau, (ndf + 3.0) * kT * tau_p * tau_p
    xi, pe = torch.zeros_like(kT), torch.zeros_like(kT)
    a3 = 1.0 + 3.0 / ndf
    f, e, w = m.evaluate(x)
    nh, npt = ensemble in ("nh", "npt"), ensemble == "npt"

    def thermostat(v, xi):
        xi = xi + dt / (4 * Q) * (2 * m.kinetic(v) - ndf * kT)
        v = v * m.per_atom(torch.exp(-0.5 * dt * xi))
        return v, xi + dt / (4 * Q) * (2 * m.kinetic(v) - ndf * kT)

    def barostat(v, pe):
        return pe + 0.5 * dt * (2 * a3 * m.kinetic(v) + w[:, :3].sum(1) - 3 * p / ATM * m.L.prod(1))

    def friction(v, pe):
        return v * m.per_atom(torch.exp(-0.5 * dt * a3 * pe / W))

    for _ in range(steps):
        if nh:
            v, xi = thermostat(v, xi)
        if npt:
            pe = barostat(v, pe)
            v = friction(v, pe)
        v = v + 0.5 * dt * FCONV / MASS * f
        if npt:
            u = dt * pe / W
            x = (x + v * dt * m.per_atom(-torch.expm1(-u) / torch.where(u == 0, torch.ones_like(u), u)
                                         + (u == 0).to(F64))) * m.per_atom(torch.exp(u))
            m.L = m.L * torch.exp(u)[:, None]
            m.x_list = None
        else:
            x = x + dt * v
        f, e, w = m.evaluate(x)
        v = v + 0.5 * dt * FCONV / MASS * f
        if npt:
            v = friction(v, pe)
            pe = barostat(v, pe)
        if nh:
            v, xi = thermostat(v, xi)
        if ensemble == "scale":
            v = v * m.per_atom(torch.sqrt(ndf * kT / (2 * m.kinetic(v))))
    return x, v, e


# ------------------------------------------------------------------ inputs


def solute_table():
    """Water (0) and a solute (1) with two-body terms only; entry (a, b, c) is the set of centre a with legs b, c."""
    t = np.zeros((2, 2, 2, 10))
    for a in range(2):
        for b in range(2):
            for c in range(2):
                e = [LAM, EPS, SIG, A_, GAM, AA, BB, C0, 4.0, 0.0]
                if a + b == 2:
                    e[1], e[2] = 0.34, 3.4
                elif a != b:
                    e[1], e[2] = 0.25, 2.88
                if a + b + c:
                    e[0] = 0.0
                    if b != c:
                        e[1] = EPS
                t[a, b, c] = e
    return t


def ice(n, rho):
    """Hexagonal ice (oxygen sites), orthorhombic cells of 8, as many as make n atoms with an edge ratio near one."""
    a = (2.0 * math.sqrt(2.0) * VMOL / rho) ** (1.0 / 3.0)
    cell = np.array([a, math.sqrt(3.0) * a, math.sqrt(8.0 / 3.0) * a])
    k = round((n / 8) ** (1.0 / 3.0))
    reps = (k, k, k)
    if 8 * k ** 3 != n:
        k = round((n / 16) ** (1.0 / 3.0))
        reps = (2 * k, k, k)
    frac = np.array([[0, 2, 0], [3, 5, 0], [3, 1, 3], [0, 4, 3], [0, 2, 2.25], [3, 5, 2.25], [3, 1, 5.25], [0, 4, 5.25]]) / 6
    g = np.stack(np.meshgrid(*[np.arange(r) for r in reps], indexing="ij"), -1).reshape(-1, 1, 3)
    return ((g + frac) * cell).reshape(-1, 3), cell * reps


def grid(rng, n, lo, ext, jitter):
    """n atoms on sites of a grid filling the region, picked at random, with a Gaussian displacement."""
    s = (np.prod(ext) / n) ** (1.0 / 3.0)
    m = [max(1, int(round(e / s))) for e in ext[:2]]
    m.append(-(-n // (m[0] * m[1])))
    g = np.stack(np.meshgrid(*[(np.arange(k) + 0.5) * e / k for k, e in zip(m, ext)], indexing="ij"), -1).reshape(-1, 3)
    pick = np.sort(rng.permutation(len(g))[:n])
    return lo + g[pick] + rng.normal(0.0, jitter, (n, 3))


def state(case, seed):
    """Positions, velocities, atoms and edges of every box, temperatures and species of a case: a function of the
    case and the seed."""
    rng = np.random.default_rng([int(seed), case["n"], case["boxes"]])
    kb, hi, lo = case["boxes"], case["n"], case.get("n_min", case["n"])
    types = None
    if case.get("system") == "slab":  # ice below, a liquid's density on a jittered grid above
        half = hi // 2
        xi, bi = ice(half, 0.92)
        lz = half * VMOL / 0.9998 / (bi[0] * bi[1])
        xl = grid(rng, half, np.array([0, 0, bi[2]]), np.array([bi[0], bi[1], lz]), 0.1)
        xs, n, L, T = [xi + rng.normal(0.0, 0.05, xi.shape), xl], [hi], [bi + [0, 0, lz]], [250.0]
    else:
        n = [int(k) for k in np.random.default_rng([hi, lo, kb]).integers(lo, hi + 1, kb)]  # the case's, whatever the seed
        scan = lo < hi
        rho = rng.uniform(0.92, 1.10, kb) if scan else np.full(kb, 0.997)
        T = list(rng.uniform(200.0, 320.0, kb)) if scan else [240.0 if case.get("ice") else 298.0] * kb
        xs, L = [], []
        for b in range(kb):
            if case.get("ice") and b == 0:
                x, box = ice(n[b], 0.92)
                x = x + rng.normal(0.0, 0.1, x.shape)
            else:
                box = np.full(3, (n[b] * VMOL / rho[b]) ** (1.0 / 3.0))
                x = grid(rng, n[b], 0.0, box, 0.1 if scan else 0.25)
            xs.append(x)
            L.append(box)
    x = torch.from_numpy(np.concatenate(xs)).cuda()
    L = np.array(L)
    if case.get("solute"):  # low density at first: the solutes are larger than water
        types = torch.from_numpy((rng.random(len(x)) < case["solute"]).astype(np.int32)).cuda()
        L = L * (1.0 + 0.45 * case["solute"])
        x = x * (1.0 + 0.45 * case["solute"])
    m = Model(n, L, None if types is None else types.long())
    sd = torch.sqrt(torch.tensor(T, dtype=F64, device="cuda") * KB / MASS * FCONV)
    v = torch.from_numpy(rng.standard_normal((len(x), 3))).cuda() * m.per_atom(sd)
    mean = torch.zeros(len(n), 3, dtype=F64, device="cuda").index_add_(0, m.bid, v) / m.n[:, None]
    v = v - mean[m.bid]
    if len(x) <= 100000:  # settle: a liquid's structure and speeds
        steps = 30 if case["kind"] != "fit" else 10
        x, v, _ = dynamics(m, x, v, steps, "scale", T, dt=8.0)
    elif case["kind"] != "md":
        x, v, _ = dynamics(m, x, v, 10, "scale", T, dt=8.0)
    lb = m.L[m.bid]
    return {"x": (x - lb * torch.floor(x / lb)).contiguous(), "v": v.contiguous(), "n": n, "L": L, "T": T,
            "types": types}


ENSEMBLE = {"nve": mw.MW_NVE, "nh": mw.MW_NOSE_HOOVER, "npt": mw.MW_NPT}
FIT_START = ((21.0, EPS * 1.05, SIG * 1.05), (21.02, EPS * 1.049, SIG * 1.0495))  # an iterate and a trial step


def system(st, case):
    s = mw.System(st["n"] if case["boxes"] > 1 else st["n"][0], st["L"] if case["boxes"] > 1 else st["L"][0],
                  skin=case.get("skin", 1.0))
    if st["types"] is not None:
        s.set_species(solute_table(), st["types"].cpu().numpy())
    if case.get("engine") == "graph":
        s.set_engine(mw.MW_ENGINE_GRAPH)
    return s


def prepare(case, seed):
    st = state(case, seed)
    p = {"case": case, "x": st["x"], "v": st["v"]}
    if case["kind"] == "fit":
        p["x"] = st["x"].float().requires_grad_()  # a torch program's dtype
        p["ff"] = torch_ops.ForceField(st["n"] if case["boxes"] > 1 else st["n"][0],
                                       st["L"] if case["boxes"] > 1 else st["L"][0])
        p["target"] = Model(st["n"], st["L"]).evaluate(p["x"].detach().double())[0].float()
        p["theta"] = [torch.tensor(t, requires_grad=True) for t in FIT_START]
        return p
    p["sys"] = system(st, case)
    if case["kind"] == "md":
        # a user keeps one integrator for a run
        p["integ"] = mw.make_integrator(dt=10.0, thermostat=ENSEMBLE[case["ensemble"]], tau=1000.0, p_ext=0.0,
                                        tau_p=2500.0, T0_per_box=st["T"])
        p["out"] = torch.empty_like(st["x"]), torch.empty_like(st["v"])
        if case["ensemble"] == "npt":
            mw.mw_set_state_dev(p["sys"].h, st["x"], st["v"])
            p["saved"] = p["sys"].checkpoint()
    elif case["kind"] == "frames":
        k, N, nb = case["frames"], len(st["x"]), case["boxes"]
        p["x"] = [st["x"]] + [state(case, seed * 16 + 5 + i)["x"] for i in range(1, k)]
        p["f"] = torch.empty(k, N, 3, dtype=torch.float32, device="cuda")
        p["e"] = torch.empty(k, nb, 3, dtype=F64, device="cuda")
        p["w"] = torch.empty(k, nb, 6, dtype=F64, device="cuda")
    return p


# ------------------------------------------------------------------ one pass


def run(p):
    case = p["case"]
    if case["kind"] == "md":
        s, (xo, vo) = p["sys"], p["out"]
        if case["ensemble"] == "npt":  # a segment from a saved state: the barostat left another box behind
            s.restore(p["saved"])
        else:
            mw.mw_set_state_dev(s.h, p["x"], p["v"])
        th = mw.mw_step(s.h, p["integ"], case["steps"], s.nbox)
        mw.mw_get_state_dev(s.h, xo, vo)
        rec = {k: [t[k] for t in th] for k in ("pe", "ke", "volume")}
        return {"x": xo, "v": vo, **(rec if s.nbox <= 16 else {k: np.array(r) for k, r in rec.items()})}
    if case["kind"] == "frames":
        for k, x in enumerate(p["x"]):
            mw.mw_energy_forces_dev(p["sys"].h, x, p["f"][k], p["e"][k], p["w"][k])
        return {"f": p["f"], "e": p["e"].float(), "w": p["w"].float()}  # labels of a training set, kept in FP32
    if case["kind"] == "fit":
        out = []
        for theta in p["theta"]:
            f = p["ff"].forces(p["x"], theta)
            gx, gt = torch.autograd.grad(torch_ops.force_matching_loss(f, p["target"]), (p["x"], theta))
            out.append({"f": f.detach(), "gx": gx, "gtheta": gt})
        return out
    s = p["sys"]
    mw.mw_set_state_dev(s.h, p["x"])
    return {"g": s.pair_histogram(0.05, int(5.8 / 0.05)).astype(np.int64),
            "adf": s.angle_histogram(8, 180).astype(np.int64)}


# ------------------------------------------------------------------ what a pass cannot do without, and what it gives


LEGS = 9.0  # ordered pairs inside the cutoff, an atom


def work(case):
    n = 0.5 * (case["n"] + case.get("n_min", case["n"])) * case["boxes"]
    # a leg's terms and its share of the angle sums and of the forces: about 190 operations
    force = n * LEGS * 190.0
    if case["kind"] == "md":
        return {"bytes": 96.0 * n, "flops": case["steps"] * (force + 60.0 * n)}
    if case["kind"] == "frames":
        return {"bytes": case["frames"] * 36.0 * n, "flops": case["frames"] * force}
    if case["kind"] == "fit":
        return {"bytes": 2 * (24.0 + 12 + 12 + 12 + 24) * n, "flops": 2 * 3.5 * force}
    return {"bytes": 24.0 * n, "flops": n * (35 * 12.0 + 28 * 30.0)}


def exact(case, seed):
    if case["kind"] == "structure":
        return None  # whole numbers
    st = state(case, seed)
    m = Model(st["n"], st["L"], None if st["types"] is None else st["types"].long())
    if case["kind"] == "md":
        x, v, e = dynamics(m, st["x"], st["v"], case["steps"], case["ensemble"], st["T"])
        lb = m.L[m.bid]
        rec = {"pe": e[:, 0].tolist(), "ke": m.kinetic(v).tolist(), "volume": m.L.prod(1).tolist()}
        return {"x": x - lb * torch.floor(x / lb), "v": v,
                **(rec if case["boxes"] <= 16 else {k: np.array(r) for k, r in rec.items()})}
    if case["kind"] == "frames":
        xs = [st["x"]] + [state(case, seed * 16 + 5 + i)["x"] for i in range(1, case["frames"])]
        out = [Model(st["n"], st["L"]).evaluate(x) for x in xs]
        return {"f": torch.stack([o[0] for o in out]), "e": torch.stack([o[1] for o in out]),
                "w": torch.stack([o[2] for o in out])}
    x32 = st["x"].float().double()
    target = m.evaluate(x32)[0].float().double()
    out = []
    for t in FIT_START:
        t = [float(np.float32(k)) for k in t]
        th = torch.tensor(t, dtype=F64, device="cuda", requires_grad=True)
        mt = Model(st["n"], st["L"], theta=t)
        mt.lam, mt.eps, mt.sig = th[0], th[1], th[2]
        x = x32.clone().requires_grad_()
        i, j = mt.legs(x32)
        d = mt.vec(x, i, j)
        e2, e3 = mt.terms(d, i, j)
        g, = torch.autograd.grad(e2.sum() + e3.sum(), d, create_graph=True)
        f = torch.zeros_like(x32).index_add(0, i, g).index_add(0, j, -g)
        gx, gt = torch.autograd.grad(((f - target) ** 2).mean(), (x, th))
        out.append({"f": f.detach(), "gx": gx, "gtheta": gt})
    return out
