"""The work a user of the library has it do, as cases that can be timed.

A case is one call sequence through the public binding
(`paper_2608_14911_gb300.espp`) on seeded synthetic inputs: integrating
Kremer-Grest melts, Lennard-Jones and DPD fluids, batches of melts and
coarse-grained melts with the learned potential, one force-matching gradient,
and the evaluation of stored frames.  `listed()` holds the named cases,
`draw(rng)` gives others of the same ranges.

A pass that integrates continues the trajectory of its handle, as a program
does that runs a few steps between two looks at the state, and returns the
whole state afterwards: unwrapped positions and velocities in the handle's own
precision (a wrapped coordinate jumps by a box edge where a rounding differs at
a face; the unwrapped one does not).  The step counts keep two passes well
inside the time over which such a system forgets the last bits of its start.

`exact(case, seed)` is the same physics in plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2608_14911_gb300 import espp, inputs

WCA_RC = 2.0 ** (1.0 / 6.0)
KG_SKIN = 0.4
MLP_RC = 3.5
FENE_K, FENE_R0 = 30.0, 1.5
DPD_A, DPD_GAMMA, DPD_DT, DPD_SKIN = 25.0, 4.5, 0.04, 0.6
DT = 0.005


def listed():
    return [
        # the first thing a new user runs: a 20 x 50 bead melt in FP64; every
        # launch and every dependent load counts
        dict(name="kg_1k_fp64", kind="kg", chains=20, beads=50, precision=64, steps=50),
        # a small production melt in FP32: still a fraction of the chip
        dict(name="kg_5k_fp32", kind="kg", chains=100, beads=50, precision=32, steps=25),
        # the large melt the package is used for: 1000 chains of 1000 beads
        dict(name="kg_1m_fp32", kind="kg", chains=1000, beads=1000, precision=32, steps=12),
        # the same melt on the reference precision
        dict(name="kg_1m_fp64", kind="kg", chains=1000, beads=1000, precision=64, steps=10),
        # a Lennard-Jones fluid of ordinary size, an odd number of unit cells
        dict(name="lj_27k_fp32", kind="lj", nx=19, ny=19, nz=19, precision=32, steps=40),
        # the largest fluid: 4.2 million atoms, long lists
        dict(name="lj_4m_fp32", kind="lj", nx=128, ny=128, nz=64, precision=32, steps=20),
        # independent melts of uneven size stepped together (parameter sweeps)
        dict(name="batch_64_fp32", kind="batch", replicas=64, size_seed=42, precision=32, steps=12),
        # a DPD fluid at rest on the Verlet list
        dict(name="dpd_786k_fp32", kind="dpd", edge=64, shear=0.0, cells=False, precision=32, steps=5),
        # a DPD fluid under Lees-Edwards shear, list-free cell forces
        dict(name="dpd_shear_24k_fp32", kind="dpd", edge=20, shear=0.01, cells=True, precision=32, steps=5),
        # a coarse-grained melt with the learned potential
        dict(name="cg_400k_mlp", kind="cg", chains=1600, beads=250, precision=32, steps=5),
        # the gradient of the force-matching loss over two mapped frames
        dict(name="fit_100k_2_frames", kind="fit", chains=2000, beads=50, frames=2),
        # a stored frame evaluated: forces, observables, distance histogram
        dict(name="frame_200k_fp32", kind="frame", chains=1000, beads=200, precision=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kg", "kg", "kg64", "lj", "lj", "batch", "dpd", "dpd_cells", "cg", "fit", "frame"])
    if kind in ("kg", "kg64"):
        m = _log_int(rng, 9, 98)
        beads = _log_int(rng, 10, min(1000, m * m))
        chains = m ** 3 // beads
        fp64 = kind == "kg64"
        steps = (50 if chains * beads < 20_000 else 10) if fp64 else (25 if chains * beads < 50_000 else 12)
        return dict(kind="kg", chains=chains, beads=beads, precision=64 if fp64 else 32, steps=steps)
    if kind == "lj":
        a = _log_int(rng, 7, 90)
        nx, ny, nz = (max(7, min(100, a + rng.randint(-a // 5, a // 5))) for _ in range(3))
        n = 4 * nx * ny * nz
        fp64 = rng.random() < 0.25 and n < 300_000
        return dict(kind="lj", nx=nx, ny=ny, nz=nz, precision=64 if fp64 else 32,
                    steps=10 if fp64 else (40 if n < 200_000 else 20))
    if kind == "batch":
        return dict(kind="batch", replicas=_log_int(rng, 2, 60), size_seed=rng.randint(1, 10_000), precision=32,
                    steps=12)
    if kind in ("dpd", "dpd_cells"):
        cells = kind == "dpd_cells"
        edge = _log_int(rng, 8, 40 if cells else 60)
        return dict(kind="dpd", edge=edge, shear=rng.choice([0.0, 0.01]), cells=cells, precision=32, steps=5)
    if kind == "cg":
        beads = rng.randint(20, 300)
        n = _log_int(rng, 5_000, 390_000)
        return dict(kind="cg", chains=max(20, n // beads), beads=beads, precision=32, steps=5)
    if kind == "fit":
        beads = rng.randint(20, 80)
        n = _log_int(rng, 5_000, 95_000)
        return dict(kind="fit", chains=max(60, n // beads), beads=beads, frames=rng.randint(1, 2))
    m = _log_int(rng, 12, 57)
    beads = _log_int(rng, 10, min(400, m * m))
    return dict(kind="frame", chains=m ** 3 // beads, beads=beads, precision=rng.choice([32, 64]))


# ---- inputs --------------------------------------------------------------------
def _melt(chains, beads, seed):
    """A melt on the lattice of a full cube at density 0.85 (1.0557 between
    neighbours whatever the bead count)."""
    n = chains * beads
    m = math.ceil(n ** (1.0 / 3.0) - 1e-9)
    return inputs.kg_lattice(chains, beads, density=0.85 * n / m ** 3, seed=seed)


def _mlp_weights():
    g = np.random.default_rng(4)
    w = np.concatenate([g.normal(0, 0.18, 64 * 32), np.zeros(64), g.normal(0, 0.125, 64 * 64), np.zeros(64),
                        g.normal(0, 0.06, 64), [0.0]])
    return espp.to_bf16_bits(w)


def _start(case, seed):
    """Configuration(s) and velocities in id order: [(Config, v, thermostat seed)]."""
    kind = case["kind"]
    if kind == "batch":
        sizes = inputs.replica_sizes(case["replicas"], seed=case["size_seed"])
        out = []
        for r, (nc, nb) in enumerate(sizes):
            c = _melt(nc, nb, seed + 1000 * r)
            out.append((c, inputs.maxwell_velocities(c.n, 1.0, seed=seed + 1000 * r), seed + r))
        return out
    if kind in ("kg", "frame"):
        c = _melt(case["chains"], case["beads"], seed)
        kT = 1.0
    elif kind == "lj":
        c = inputs.lj_fcc(case["nx"], case["ny"], case["nz"], density=0.8442)
        g = np.random.default_rng(seed)
        c.x = inputs.f32(np.mod(c.x + g.uniform(-0.06, 0.06, c.x.shape), c.box))
        c.x[c.x >= c.box] = 0.0
        kT = 0.72
    elif kind == "dpd":
        e = float(case["edge"])
        c = inputs.random_positions(3 * case["edge"] ** 3, (e, e, e), seed=seed)
        kT = 1.0
    else:  # cg, fit
        c = inputs.kg_lattice(case["chains"], case["beads"], density=0.2125, seed=seed, jitter=0.3)
        kT = 1.0
    return [(c, inputs.maxwell_velocities(c.n, kT, seed=seed), seed)]


def _fit_frames(case, c, seed):
    """Mapped frames and their target forces, (frames, n, 3) on the GPU."""
    g = np.random.default_rng(seed)
    X = np.stack([inputs.f32(np.mod(c.x + g.normal(0, 0.2, c.x.shape), c.box)) for _ in range(case["frames"])])
    X[X >= c.box] = 0.0
    return torch.tensor(X, device="cuda"), torch.tensor(g.normal(0, 1.0, X.shape), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    start = _start(case, seed)
    prec = espp.ESPP_FP64 if case.get("precision") == 64 else espp.ESPP_FP32
    types = [None if kind in ("cg", "fit", "dpd") else c.types for c, _, _ in start]
    s = espp.System(precision=prec, replicas=[
        dict(box=c.box, n=c.n, types=t, bonds=c.bonds, seed=sd) for (c, _, sd), t in zip(start, types)])
    x = torch.tensor(np.concatenate([c.x for c, _, _ in start]), device="cuda")
    v = torch.tensor(np.concatenate([v for _, v, _ in start]), device="cuda")
    img = torch.tensor(np.concatenate([c.img for c, _, _ in start]), device="cuda")
    st = dict(case=case, s=s, x=x, v=v, img=img,
              real=torch.float64 if prec == espp.ESPP_FP64 else torch.float32,
              box=torch.tensor(np.concatenate([np.broadcast_to(c.box, (c.n, 3)) for c, _, _ in start])
                               if len(start) > 1 else start[0][0].box, device="cuda"))
    if kind in ("kg", "batch", "frame"):
        s.set_wca()
        s.set_fene(FENE_K, FENE_R0)
        st["run"] = (DT, 1.0, 1.0)
        rc, skin = WCA_RC, KG_SKIN
    elif kind == "lj":
        s.set_lj(1.0, 1.0, 2.5, True)
        st["run"] = (DT, 1.0, 0.72)
        rc, skin = 2.5, 0.3
    elif kind == "dpd":
        r = np.linspace(0.0, 1.0, 1001)
        s.set_table_pair(1.0, 0.5 * DPD_A * (1.0 - r) ** 2, DPD_A * (1.0 - r))
        s.set_thermostat(espp.ESPP_THERMO_DPD, 1.0)
        if case["shear"]:
            s.set_lees_edwards(True, case["shear"], 0.0)
        if case["cells"]:
            s.set_force_method(espp.ESPP_FORCES_CELLS)
        st["run"] = (DPD_DT, DPD_GAMMA, 1.0)
        rc, skin = 1.0, DPD_SKIN
    else:
        s.set_mlp(MLP_RC, _mlp_weights())
        rb = np.linspace(0.0, 6.0, 1201)
        s.set_table_bond(6.0, 2.0 * (rb - 2.0) ** 2, -4.0 * (rb - 2.0))
        s.set_exclude_bonded(True)
        st["run"] = (DT, 1.0, 1.0)
        rc, skin = MLP_RC, 0.5 if kind == "cg" else 0.0
    s.set_state(x, v, img)
    s.build_neighbors(rc, skin)
    if kind == "fit":
        st["X"], st["Y"] = _fit_frames(case, start[0][0], seed)
    else:
        st["out"] = (torch.empty_like(x), torch.empty_like(v), torch.empty_like(img))
        st["f"] = torch.empty_like(x)
    return st


OBS = ("ke", "pe_pair", "pe_bond", "virial", "temperature", "pressure", "mean_bond", "rg2")
RDF_MAX, RDF_BINS = 1.5, 150


def run(st):
    case, s = st["case"], st["s"]
    if case["kind"] == "fit":
        loss, grad = s.mlp_loss_grad(st["X"], st["Y"])
        return {"loss": loss, "grad": grad.astype(np.float32)}  # the library's gradient is FP32
    if case["kind"] == "frame":
        s.set_state(st["x"], st["v"], st["img"])
        s.compute_forces(st["f"])
        o = s.observables()
        counts = s.rdf_counts(RDF_MAX, RDF_BINS)
        return {"forces": st["f"].to(st["real"]), "observables": [o[k] for k in OBS], "counts": counts}
    s.integrate(case["steps"], *st["run"])
    x, v, img = s.get_state(st["out"])
    u = torch.addcmul(x, img, st["box"])
    if case.get("shear"):
        # the image above a sheared face is displaced and moving
        _, rate, t = s.lees_edwards()
        top = rate * float(case["edge"])
        u[:, 0] += img[:, 2] * (top * t)
        v = v.clone()
        v[:, 0] += img[:, 2] * top
    return {"positions": u.to(st["real"]), "velocities": v.to(st["real"])}


# ---- what a pass cannot do without ----------------------------------------------
def _count(case):
    kind = case["kind"]
    if kind == "lj":
        return 4 * case["nx"] * case["ny"] * case["nz"]
    if kind == "dpd":
        return 3 * case["edge"] ** 3
    if kind == "batch":
        return sum(a * b for a, b in inputs.replica_sizes(case["replicas"], seed=case["size_seed"]))
    return case["chains"] * case["beads"]


def work(case):
    kind, n = case["kind"], _count(case)
    real = 8 if case.get("precision") == 64 else 4
    sphere = 4.0 / 3.0 * math.pi
    if kind in ("kg", "batch", "frame"):
        pairs, per_pair, other = 0.85 * sphere * WCA_RC ** 3 / 2, 40, 100  # FENE, thermostat, integration
    elif kind == "lj":
        pairs, per_pair, other = 0.8442 * sphere * 2.5 ** 3 / 2, 30, 50
    elif kind == "dpd":
        pairs, per_pair, other = 3.0 * sphere / 2, 150, 20  # the pair's Philox draw included
    else:
        pairs, per_pair, other = 0.2125 * sphere * MLP_RC ** 3 / 2, 24576, 100
    if kind == "fit":
        # forward values and tangents, then the reverse pass to the weights
        return {"bytes": case["frames"] * n * 48 + 2 * 4 * 6336,
                "flops": case["frames"] * n * (pairs * 3 * per_pair + other)}
    if kind == "frame":
        return {"bytes": n * (9 * 8 + 12 + 6 * real), "flops": n * (pairs * per_pair + other)}
    # positions and velocities read and written once a step
    return {"bytes": case["steps"] * n * 12 * real, "flops": case["steps"] * n * (pairs * per_pair + other)}


# ---- the same in 64 bits ----------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
    return c0, c1, c2, c3


def _centred(w):
    return (2 * (w >> 8) + 1 - 16777216).double() * 2.0 ** -25


class _Exact:
    """One system in 64 bits: unwrapped positions, unordered pair list with a
    skin, forces, velocity Verlet."""

    def __init__(self, case, c, v, seed):
        self.case, self.seed, self.n = case, seed, c.n
        self.box = torch.tensor(c.box, device="cuda")
        self.u = torch.tensor(c.x, device="cuda") + torch.tensor(c.img, device="cuda") * self.box
        self.v = torch.tensor(v, device="cuda")
        self.b = torch.tensor(c.bonds, device="cuda") if len(c.bonds) else None
        self.id = torch.arange(c.n, device="cuda")
        self.shear = case.get("shear") or 0.0
        self.rc = {"lj": 2.5, "dpd": 1.0, "cg": MLP_RC, "fit": MLP_RC}.get(case["kind"], WCA_RC)
        self.built = None
        if case["kind"] in ("cg", "fit"):
            w = torch.tensor(espp.bf16_bits_to_float(_mlp_weights()), device="cuda")
            sizes = [64 * 32, 64, 64 * 64, 64, 64]
            W1, b1, W2, b2, w3 = (p.clone() for p in torch.split(w[:-1], sizes))
            self.net = [W1.view(64, 32), b1, W2.view(64, 64), b2, w3]

    # -- geometry
    def offset(self, t):
        return self.shear * float(self.box[2]) * t

    def separation(self, i, j, t):
        d = self.u[i] - self.u[j]
        nz = torch.round(d[:, 2] / self.box[2])
        d[:, 0] -= nz * self.offset(t)
        d -= self.box * torch.round(d / self.box)
        return d, nz

    def pairs(self, t, skin=0.3):
        if self.built is not None and 2 * float((self.u - self.built).norm(dim=1).max()) + abs(
                self.offset(t) - self.off0) < skin:
            return self.ij
        self.built, self.off0 = self.u.clone(), self.offset(t)
        rl = self.rc + skin
        # cells in the coordinates of the (possibly sheared) box
        f = self.u / self.box
        f[:, 0] -= torch.floor(f[:, 2]) * self.off0 / self.box[0] + (f[:, 2] - torch.floor(f[:, 2])) * self.off0 / self.box[0]
        f = f - torch.floor(f)
        tilt = math.sqrt(1 + (self.off0 / float(self.box[2])) ** 2)
        nc = [max(1, int(float(L) / (rl * tilt))) for L in self.box]
        if min(nc) < 3:
            i, j = torch.triu_indices(self.n, self.n, 1, device="cuda")
            return self.keep(i, j, t, rl)
        cell = [torch.clamp((f[:, k] * nc[k]).long(), max=nc[k] - 1) for k in range(3)]
        key = (cell[2] * nc[1] + cell[1]) * nc[0] + cell[0]
        order = torch.argsort(key)
        count = torch.bincount(key, minlength=nc[0] * nc[1] * nc[2])
        first = torch.cumsum(count, 0) - count
        rank = torch.empty_like(order)
        rank[order] = torch.arange(self.n, device="cuda")
        got = []
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    if (dz, dy, dx) < (0, 0, 0):
                        continue
                    k2 = (((cell[2] + dz) % nc[2]) * nc[1] + (cell[1] + dy) % nc[1]) * nc[0] + (cell[0] + dx) % nc[0]
                    m = count[k2]
                    i = torch.repeat_interleave(self.id, m)
                    at = torch.arange(i.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
                    at += first[k2][i]
                    j = order[at]
                    if (dz, dy, dx) == (0, 0, 0):
                        ok = at > rank[i]
                        i, j = i[ok], j[ok]
                    got.append(self.keep(i, j, t, rl))
        self.ij = torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
        return self.ij

    def keep(self, i, j, t, rl):
        out = []
        for a in range(0, i.numel(), 1 << 26):
            p, q = i[a:a + (1 << 26)], j[a:a + (1 << 26)]
            d, _ = self.separation(p, q, t)
            ok = (d * d).sum(1) < rl * rl
            if self.case["kind"] in ("cg", "fit"):  # chain neighbours feel the bond only
                nb = self.case["beads"]
                ok &= ~(((p - q).abs() == 1) & (p // nb == q // nb))
            out.append((p[ok], q[ok]))
        self.ij = torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])
        return self.ij

    # -- the learned potential: u and du/dr
    def mlp(self, r):
        W1, b1, W2, b2, w3 = self.net
        w = MLP_RC / 31
        d = r[:, None] - w * torch.arange(32, device="cuda")
        g = torch.exp(-d * d / (2 * w * w))
        fc = 0.5 * (torch.cos(math.pi * r / MLP_RC) + 1)[:, None]
        dfc = -0.5 * math.pi / MLP_RC * torch.sin(math.pi * r / MLP_RC)[:, None]
        h, dh = g * fc, g * (dfc - d / (w * w) * fc)
        for W, b in ((W1, b1), (W2, b2)):
            z, dz = h @ W.T + b, dh @ W.T
            s = torch.sigmoid(z)
            h, dh = z * s, s * (1 + z * (1 - s)) * dz
        return dh @ w3

    # -- conservative pair force over distance; energy
    def pair(self, r2):
        kind = self.case["kind"]
        if kind == "dpd":
            r = r2.sqrt()
            return DPD_A * (1 - r) / r, 0.5 * DPD_A * (1 - r) ** 2
        if kind in ("cg", "fit"):
            r = r2.sqrt()
            out = torch.cat([-self.mlp(q) / q for q in torch.split(r, 1 << 19)]) if r.numel() else r
            return out, torch.zeros_like(r)
        x = 1 / r2
        s6 = x * x * x
        c6 = self.rc ** -6
        return 24 * s6 * (2 * s6 - 1) * x, 4 * s6 * (s6 - 1) - 4 * c6 * (c6 - 1)

    def forces(self, t, thermostat=None, step=0):
        """Total force; thermostat: (gamma, kT, dt) or None."""
        f = torch.zeros_like(self.u)
        self.pe = self.vir = 0.0
        dpd = thermostat is not None and self.case["kind"] == "dpd"
        i_all, j_all = self.pairs(t)
        for a in range(0, i_all.numel(), 1 << 25):
            i, j = i_all[a:a + (1 << 25)], j_all[a:a + (1 << 25)]
            d, nz = self.separation(i, j, t)
            r2 = (d * d).sum(1)
            ok = r2 < self.rc * self.rc
            i, j, d, nz, r2 = i[ok], j[ok], d[ok], nz[ok], r2[ok]
            fr, u = self.pair(r2)
            if dpd:
                gamma, kT, dt = thermostat
                r = r2.sqrt()
                w = 1 - r
                dv = self.v[i] - self.v[j]
                dv[:, 0] -= nz * self.shear * self.box[2]
                lo, hi = torch.minimum(i, j), torch.maximum(i, j)
                th = _centred(_philox(lo, hi | 0x80000000, torch.full_like(lo, step & _M32),
                                      torch.full_like(lo, step >> 32), self.seed)[0])
                ev = (d * dv).sum(1) / r
                fr = fr + (-gamma * w * w * ev + math.sqrt(24 * gamma * kT / dt) * w * th) / r
            self.pe += float(u.sum())
            self.vir += float((fr * r2).sum())
            q = fr[:, None] * d
            f.index_add_(0, i, q)
            f.index_add_(0, j, -q)
        if self.b is not None:
            i, j = self.b[:, 0], self.b[:, 1]
            d, _ = self.separation(i, j, t)
            r2 = (d * d).sum(1)
            if self.case["kind"] in ("cg", "fit"):
                fr = -4.0 * (r2.sqrt() - 2.0) / r2.sqrt()
            else:
                m = 1 - r2 / FENE_R0 ** 2
                fr = -FENE_K / m
                self.pe_bond = float((-0.5 * FENE_K * FENE_R0 ** 2 * torch.log(m)).sum())
                self.mean_bond = float(r2.sqrt().mean())
            self.vir += float((fr * r2).sum())
            q = fr[:, None] * d
            f.index_add_(0, i, q)
            f.index_add_(0, j, -q)
        if thermostat is not None and not dpd:
            gamma, kT, dt = thermostat
            z = torch.zeros_like(self.id)
            w = _philox(self.id, z + (step & _M32), z + (step >> 32), z, self.seed)
            f += -gamma * self.v + math.sqrt(24 * gamma * kT / dt) * torch.stack([_centred(k) for k in w[:3]], 1)
        return f

    def integrate(self, steps, dt, gamma, kT):
        f = self.forces(0.0, (gamma, kT, dt), 0)
        for s in range(1, steps + 1):
            self.v += 0.5 * dt * f
            self.u += dt * self.v
            f = self.forces(s * dt, (gamma, kT, dt), s)
            self.v += 0.5 * dt * f


def exact(case, seed):
    kind = case["kind"]
    start = _start(case, seed)
    if kind == "fit":
        return _exact_fit(case, start[0][0], seed)
    if kind == "frame":
        c, v, sd = start[0]
        e = _Exact(case, c, v, sd)
        f = e.forces(0.0)
        ke = float(0.5 * (e.v * e.v).sum())
        vol = float(e.box.prod())
        x = e.u.view(case["chains"], case["beads"], 3)
        rg2 = float(((x - x.mean(1, keepdim=True)) ** 2).sum(2).mean())
        obs = [ke, e.pe, e.pe_bond, e.vir, 2 * ke / (3 * e.n), (2 * ke + e.vir) / (3 * vol), e.mean_bond, rg2]
        return {"forces": f, "observables": obs, "counts": None}
    dt, gamma, kT = {"lj": (DT, 1.0, 0.72), "dpd": (DPD_DT, DPD_GAMMA, 1.0)}.get(kind, (DT, 1.0, 1.0))
    out = []
    for c, v, sd in start:
        e = _Exact(case, c, v, sd)
        e.integrate(case["steps"], dt, gamma, kT)
        out.append((e.u, e.v))
    return {"positions": torch.cat([o[0] for o in out]), "velocities": torch.cat([o[1] for o in out])}


def _exact_fit(case, c, seed):
    X, Y = _fit_frames(case, c, seed)
    nf = case["frames"]
    loss, grad = 0.0, None
    for k in range(nf):
        e = _Exact(case, c, np.zeros((c.n, 3)), seed)
        e.u = X[k].clone()
        err = e.forces(0.0) - Y[k]
        loss += float((err * err).sum()) / (nf * c.n)
        i, j = e.pairs(0.0)
        d, _ = e.separation(i, j, 0.0)
        r = d.norm(dim=1)
        ok = r < MLP_RC
        i, j, d, r = i[ok], j[ok], d[ok], r[ok]
        w = -2.0 / (nf * c.n) * ((err[i] - err[j]) * d).sum(1) / r
        for p in e.net:
            p.requires_grad_(True)
        for rk, wk in zip(torch.split(r, 1 << 18), torch.split(w, 1 << 18)):
            (wk * e.mlp(rk)).sum().backward()
        g = torch.cat([p.grad.reshape(-1) for p in e.net])
        grad = g if grad is None else grad + g
    return {"loss": loss, "grad": grad}
