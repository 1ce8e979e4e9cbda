"""What is measured of this library's speed: the calls its users' programs make.

The cases cover the public entry points of ``paper_2002_07109_gb300.bounce``
over the range of systems that the configurations, tests and the benchmark of
this repository use:

  run      advancing a trajectory (``Context.run``) and taking one frame of it,
           for the integrators, splits and boundary conditions in use (24 steps
           between frames, the benchmark's windows);
  batch    the same for a batch of independent replicas;
  jump     one jump half-step alone (``bounce_jump_half``);
  forces   gradients at given positions (an external optimiser or driver);
  observe  energies and pair-distance histograms of stored frames;
  match    one force-matching evaluation with its backward pass;
  energy   the allocation-free pair energies.

Inputs: flexible water at 1 g/cm^3 with the repository's force field.  A
small periodic cell is relaxed from the lattice by a short Langevin run in
plain torch (no code of the library), tiled to the size of the case, and given
fresh Maxwell-Boltzmann velocities, all from the seed.

Trajectory frames and forces are returned in single precision: the library
sums the pair terms in FP32 (its FP64 output arrays carry no more than that),
and it is how trajectory files hold them.
"""
import functools
import math

import numpy as np
import torch

from paper_2002_07109_gb300 import bounce
from paper_2002_07109_gb300 import water

KCOUL, KB, ACCEL = 332.063713, 0.0019872041, 4.184e-4
BETA = 0.35                     # Ewald splitting of the boxes (1/A)
DEV = torch.device("cuda", 0)

# Bounds of a drawn batch of replicas: its atoms, and three times its molecule pairs.
BATCH_ATOMS, BATCH_PAIRS = 110000, 70000000


def listed():
    return [
        # the paper's smallest system: 64 molecules, all pairs, Coulomb and LJ on the jumps (the
        # default split); a short trajectory from a given state each time, since this split heats
        # flexible water; launches and latency decide
        {"name": "run_droplet_64", "kind": "run", "mol": 64, "n_side": 0, "integ": "BOUNCE", "coul": True, "dt": 0.25,
         "r_cut": 0.0, "steps": 64},
        # a droplet of the size of the paper's, cutoff and cell lists, LJ on the jumps
        {"name": "run_droplet_4096", "kind": "run", "mol": 4096, "n_side": 0, "integ": "BOUNCE", "coul": False, "dt": 1.0,
         "r_cut": 12.0, "steps": 24},
        # a periodic box of protein-solvent size with the three-level splitting
        {"name": "run_box_16_respa1", "kind": "run", "mol": 0, "n_side": 16, "integ": "BOUNCE_RESPA1", "coul": False,
         "dt": 1.0, "r_cut": 9.0, "steps": 24},
        # the benchmark's headline box, BOUNCE-RESPA and the BAOAB it is compared with
        {"name": "run_box_32_respa", "kind": "run", "mol": 0, "n_side": 32, "integ": "BOUNCE_RESPA", "coul": False,
         "dt": 1.0, "r_cut": 9.0, "steps": 24},
        {"name": "run_box_32_baoab", "kind": "run", "mol": 0, "n_side": 32, "integ": "BAOAB", "coul": False, "dt": 1.0,
         "r_cut": 9.0, "steps": 24},
        # many independent droplets of 64-1,024 molecules in one context
        {"name": "run_batch_64", "kind": "batch", "replicas": 64, "lo": 64, "hi": 1024, "steps": 8},
        # the jump half-step with Coulomb on the jumps (about a million proposals)
        {"name": "jump_droplet_4096", "kind": "jump", "mol": 4096, "r_cut": 12.0},
        # forces at positions given by another program: a ragged box
        {"name": "forces_box_21", "kind": "forces", "n_side": 21, "r_cut": 9.0},
        # analysis of stored frames: energies and the three radial distribution functions
        {"name": "observe_box_16", "kind": "observe", "n_side": 16, "r_cut": 9.0},
        # force matching on the 4,096-molecule box, and on the small one that fits are tried on
        {"name": "match_box_16", "kind": "match", "n_side": 16, "r_cut": 9.0},
        {"name": "match_box_6", "kind": "match", "n_side": 6, "r_cut": 9.0},
        # pair energies of a caller that cannot allocate
        {"name": "energy_droplet_1500", "kind": "energy", "mol": 1500, "n_side": 0, "r_cut": 0.0},
    ]


# Box edges in molecules that a cell of 6 to 11 molecules tiles.
SIDES = (6, 7, 8, 9, 10, 11, 12, 14, 16, 18, 20, 21, 22, 24, 27, 28, 30, 32)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def side(lo, hi):
        x = rng.uniform(math.log(lo), math.log(hi))
        return min((s for s in SIDES if lo <= s <= hi), key=lambda s: abs(math.log(s) - x))

    kind = rng.choice(("droplet", "cut", "box", "box", "box", "batch", "jump", "forces", "observe", "match", "match", "energy"))
    if kind == "droplet":       # all pairs, no cutoff
        coul = rng.random() < 0.5
        return {"kind": "run", "mol": log_int(27, 600), "n_side": 0, "integ": "BOUNCE" if coul else rng.choice(("BOUNCE", "BAOAB")),
                "coul": coul, "dt": 0.25 if coul else 1.0, "r_cut": 0.0, "steps": rng.choice((33, 48, 64))}
    if kind == "cut":
        return {"kind": "run", "mol": log_int(500, 8000), "n_side": 0, "integ": rng.choice(("BOUNCE", "BAOAB")), "coul": False,
                "dt": 1.0, "r_cut": rng.choice((9.0, 10.0, 12.0)), "steps": rng.choice((12, 24, 36))}
    if kind == "box":
        return {"kind": "run", "mol": 0, "n_side": side(8, 30), "integ": rng.choice(("BOUNCE", "BOUNCE_RESPA", "BOUNCE_RESPA1", "BAOAB")),
                "coul": False, "dt": 1.0, "r_cut": rng.choice((8.0, 9.0)), "steps": rng.choice((12, 18, 24))}
    if kind == "batch":
        lo = log_int(30, 200)
        hi = lo + log_int(16, 800)
        most = min(BATCH_ATOMS // (3 * (lo + hi) // 2), BATCH_PAIRS // (lo * lo + lo * hi + hi * hi))
        return {"kind": "batch", "replicas": log_int(2, max(2, most)), "lo": lo, "hi": hi, "steps": rng.choice((4, 8))}
    if kind == "jump":
        return {"kind": "jump", "mol": log_int(300, 4096), "r_cut": rng.choice((9.0, 10.0, 12.0))}
    if kind in ("forces", "observe"):
        return {"kind": kind, "n_side": side(7, 24), "r_cut": round(rng.uniform(8.0, 9.5), 2)}
    if kind == "match":
        return {"kind": "match", "n_side": side(6, 20), "r_cut": round(rng.uniform(7.5, 9.2), 2)}
    if rng.random() < 0.6:
        return {"kind": "energy", "mol": log_int(30, 5000), "n_side": 0, "r_cut": 0.0}
    return {"kind": "energy", "mol": 0, "n_side": side(6, 16), "r_cut": round(rng.uniform(7.5, 9.2), 2)}


# ------------------------------------------------------------------ inputs
def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(dtype)


def _pair(r2, qq, c12, c6, beta):
    """W(r) Coulomb and LJ parts and W'(r)/r of the pairs at squared distances r2 (qq holds k q_i q_j)."""
    r = r2.sqrt()
    ir2 = 1.0 / r2
    if beta > 0:
        e = torch.erfc(beta * r)
        wc = qq * e / r
        g = -qq * (e / r + 2.0 * beta / math.sqrt(math.pi) * torch.exp(-(beta * beta) * r2)) * ir2
    else:
        wc = qq / r
        g = -wc * ir2
    ir6 = ir2 * ir2 * ir2
    return wc, (c12 * ir6 - c6) * ir6, g - (12.0 * c12 * ir6 - 6.0 * c6) * ir6 * ir2


def _bonded(q, s):
    """Bond and angle energies and their gradient."""
    b, a = _t(s.bonds, torch.int64), _t(s.angles, torch.int64)
    kb, ka = _t(s.bond_k_r0, q.dtype), _t(s.angle_k_t0, q.dtype)
    g = torch.zeros_like(q)
    d = q[b[:, 0]] - q[b[:, 1]]
    r = d.norm(dim=1)
    x = r - kb[:, 1]
    f = (2.0 * kb[:, 0] * x / r)[:, None] * d
    u, w = q[a[:, 0]] - q[a[:, 1]], q[a[:, 2]] - q[a[:, 1]]
    nu, nw = u.norm(dim=1, keepdim=True), w.norm(dim=1, keepdim=True)
    cs = ((u * w).sum(1, keepdim=True) / (nu * nw)).clamp(-1.0, 1.0)
    th = torch.acos(cs) - ka[:, 1:]
    fa = -2.0 * ka[:, :1] * th / (1.0 - cs * cs).clamp_min(1e-12).sqrt()
    ga, gc = fa * (w / (nu * nw) - cs * u / nu ** 2), fa * (u / (nu * nw) - cs * w / nw ** 2)
    # every atom has its place in a fixed order: O 3m, H 3m + 1, H 3m + 2, bonds (O, H1), (O, H2), one angle
    f = f.reshape(-1, 2, 3)
    g[0::3] = f[:, 0] + f[:, 1] - ga - gc
    g[1::3] = ga - f[:, 0]
    g[2::3] = gc - f[:, 1]
    return (kb[:, 0] * x * x).sum(), (ka[:, :1] * th * th).sum(), g


@functools.lru_cache(maxsize=24)
def _cell(m, seed):
    """Positions [m^3, 3 atoms, 3] of a relaxed periodic cell of m^3 molecules: 250 steps of 1 fs from the lattice
    at friction 0.08/fs, direct-space pair terms within 9 A, in FP32."""
    s = water.water_box(m, seed=seed)
    L = float(s.box[0])
    q, v = _t(s.q, torch.float32), _t(s.v, torch.float32)
    mol, ch = _t(s.molecule, torch.int64), _t(s.charge, torch.float32)
    o = _t(s.type, torch.int64) == 0
    keep = mol[:, None] != mol[None, :]
    qq = KCOUL * ch[:, None] * ch[None, :]
    s6 = 3.15 ** 6
    oo = (o[:, None] & o[None, :]).float()
    c12, c6 = oo * (4 * 0.152 * s6 * s6), oo * (4 * 0.152 * s6)
    im = ACCEL / _t(s.mass, torch.float32)[:, None]
    c1 = math.exp(-0.08)
    sd = ((1.0 - c1 * c1) * KB * 300.0 * im).sqrt()
    gen = torch.Generator(device=DEV).manual_seed(seed % (1 << 31) + 17)
    rc = min(9.0, 0.499 * L)
    for _ in range(250):
        d = q[:, None, :] - q[None, :, :]
        d -= L * (d / L).round()
        r2 = (d * d).sum(2)
        inside = keep & (r2 < rc * rc)
        _, _, g = _pair(torch.where(inside, r2, 1.0), qq, c12, c6, BETA)
        grad = (torch.where(inside, g, 0.0)[:, :, None] * d).sum(1) + _bonded(q, s)[2]
        v = c1 * (v - (im * grad).clamp(-0.02, 0.02)) + sd * torch.randn(q.shape, generator=gen, device=DEV)
        q = q + v
    return q.double().cpu().numpy().reshape(-1, 3, 3)


def _tile_side(n):
    return next(m for m in (8, 9, 10, 7, 11, 6) if n % m == 0)


def _sites(cell, m, ijk, a):
    """The molecules of the tiled cell at the lattice sites ijk."""
    c = ((ijk[:, 0] % m) * m + ijk[:, 1] % m) * m + ijk[:, 2] % m
    return (cell[c] + (ijk // m * (m * a))[:, None, :]).reshape(-1, 3)


def _box(n, seed):
    s = water.water_box(n, seed=seed)
    m = _tile_side(n)
    g = np.arange(n)
    ijk = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    s.q = _sites(_cell(m, seed), m, ijk, water.lattice_spacing())
    return s


def _droplet(n_mol, seed, piece=0):
    """The n_mol molecules nearest the centre of a piece of the tiled cell."""
    s = water.water_droplet_molecules(n_mol, seed=seed + 1000 * piece)
    side = int(math.ceil(n_mol ** (1.0 / 3.0))) + 1
    g = np.arange(side)
    ijk = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    d2 = ((ijk - ijk.mean(0)) ** 2).sum(1)
    keep = np.sort(np.lexsort((np.arange(len(ijk)), d2))[:n_mol])
    s.q = _sites(_cell(8, seed), 8, ijk[keep] + np.array([piece % 8, piece // 8 % 8, 0]), water.lattice_spacing())
    return s


def _grid(n):
    """SPME points per edge: the next product of 2, 3 and 5 at or above three per molecule."""
    k = 3 * n
    while True:
        r = k
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1:
            return k
        k += 1


def _system(case, seed):
    return _box(case["n_side"], seed) if case.get("n_side") else _droplet(case["mol"], seed)


def _batch(case, seed):
    sizes = water.replica_sizes(case["replicas"], lo=case["lo"], hi=case["hi"], seed=case["replicas"])
    return water.concat_systems([_droplet(int(m), seed, r) for r, m in enumerate(sizes)])


def _config(case):
    """The context options of a case: the benchmark's for boxes, the paper's switch for droplets."""
    kind = case["kind"]
    if kind == "match":
        return dict(r_on=4.0, r_off=5.0, r_cut=case["r_cut"], ewald_beta=BETA, skin=1.0, max_neighbors=1024)
    if kind in ("forces", "observe"):
        return dict(r_on=case["r_cut"] - 1.5, r_off=case["r_cut"] - 0.5, r_cut=case["r_cut"], skin=1.0, pair_skin=3.0, ewald_beta=BETA, jump_coulomb=False,
                    pme_grid=(_grid(case["n_side"]),) * 3, max_neighbors=1024)
    if kind == "batch":
        return dict(r_on=4.0, r_off=5.0, jump_coulomb=False, max_neighbors=3 * case["hi"])
    if kind == "jump":
        return dict(r_on=4.0, r_off=5.0, r_cut=case["r_cut"], skin=1.0)
    c = dict(dt=case["dt"], jump_coulomb=case["coul"], respa_m=2, respa_m2=3, seed=7)
    if case["n_side"]:
        rc = case["r_cut"]
        c.update(r_on=rc - 1.5, r_off=rc - 0.5, r_cut=rc, pair_skin=3.0, ewald_beta=BETA, pme_grid=(_grid(case["n_side"]),) * 3)
        c.update(dict(skin=1.0, max_neighbors=1024) if case["integ"] == "BAOAB" else dict(skin=2.5, max_neighbors=2048))
    else:
        c.update(r_on=4.0, r_off=5.0, r_cut=case["r_cut"] or math.inf, skin=1.0)
    return c


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        s, off = _batch(case, seed)
        ctx = bounce.from_system(s, seed=1, **_config(case))
        ctx.set_replicas(off, np.arange(len(off) - 1, dtype=np.uint64) + 7)
    else:
        s = _system(case, seed)
    n = s.n_atoms
    if kind == "energy":
        st = dict(kind=kind, q=_t(s.q), charge=_t(s.charge), type=_t(s.type, torch.int32), molecule=_t(s.molecule, torch.int32),
                  sigma=s.lj_sigma, eps=s.lj_eps, out=torch.zeros(2, dtype=torch.float64, device=DEV))
        st.update(dict(box=s.box, r_cut=case["r_cut"], beta=BETA) if case["n_side"] else dict(box=None, r_cut=math.inf, beta=0.0))
        return st
    if kind != "batch":
        ctx = bounce.from_system(s, **_config(case))
    st = dict(kind=kind, ctx=ctx)
    if kind in ("forces", "observe"):
        # two frames far enough apart that nothing built for one serves the other
        shift = np.random.default_rng(seed + 5).uniform(3.0, 9.0, 3)
        st["frames"] = [(_t(s.q), _t(s.v)), (_t(s.q + shift), _t(s.v))]
    if kind == "forces":
        st["grad"] = [torch.empty((n, 3), dtype=torch.float64, device=DEV) for _ in range(4)]
        return st
    if kind == "observe":
        return st
    ctx.set_state(s.q, s.v)
    if kind == "match":
        p = _match_params(requires_grad=True)
        st.update(q=_t(s.q).requires_grad_(True), params=p, fn=bounce.pair_forces_function(), target=_match_target(s, case["r_cut"]))
        return st
    st.update(q=torch.empty((n, 3), dtype=torch.float64, device=DEV), v=torch.empty((n, 3), dtype=torch.float64, device=DEV),
              steps=case.get("steps"), step=0, start=(_t(s.q), _t(s.v)) if case.get("coul") else None, integ=getattr(bounce, case.get("integ", "BOUNCE")))
    return st


def run(st):
    kind = st["kind"]
    if kind in ("run", "batch"):
        ctx = st["ctx"]
        if st["start"] is not None:
            ctx.set_state(*st["start"])
        ctx.run(st["steps"], st["integ"])
        ctx.get_state(st["q"], st["v"])
        return {"q": st["q"].float(), "v": st["v"].float()}
    if kind == "jump":
        ctx = st["ctx"]
        m, acc = ctx.jump_half(st["step"], 1)
        st["step"] += 1
        ctx.get_state(st["q"], st["v"])
        return {"proposals": m, "accepts": acc, "v": st["v"].float()}
    if kind == "forces":
        ctx, out = st["ctx"], []
        for k, (q, v) in enumerate(st["frames"]):
            ctx.set_state(q, v)
            for part, g in ((bounce.GRAD_FULL, st["grad"][2 * k]), (bounce.GRAD_RECIP, st["grad"][2 * k + 1])):
                r = bounce.bounce_compute_gradient(ctx.h, part, g.data_ptr(), bounce.DEVICE, None)
                if r != bounce.OK:
                    raise RuntimeError("bounce_compute_gradient: %d" % r)
                out.append(g.float())
        return out
    if kind == "observe":
        ctx, out = st["ctx"], []
        for q, v in st["frames"]:
            ctx.set_state(q, v)
            e = ctx.energies()
            out.append({k: e[k] for k in ("coulomb", "lj", "bond", "angle", "kinetic", "recip", "potential")})
            out.append([ctx.pair_histogram(a, b, 8.0, 160) for a, b in ((0, 0), (0, 1), (1, 1))])
        return out
    if kind == "match":
        f, e = st["fn"].apply(st["q"], *st["params"], st["ctx"])
        loss = ((f - st["target"]) ** 2).sum()
        g = torch.autograd.grad(loss, [st["q"], *st["params"]])
        return {"forces": f.detach().float(), "energy": e.detach().float(), "loss": loss.detach().float(), "grads": [x.float() for x in g]}
    r = bounce.pair_energy_noalloc(st["q"], st["charge"], st["type"], st["molecule"], st["sigma"], st["eps"], r_cut=st["r_cut"],
                                   ewald_beta=st["beta"], box=st["box"], out=st["out"])
    if r != bounce.OK:
        raise RuntimeError("pair_energy_noalloc: %d" % r)
    return st["out"].float()


# -------------------------------------------------------------------- work
def _pairs_in(n, r_cut):
    """Pairs of different molecules within r_cut of n atoms at the density of water."""
    rho = 3.0 / water.lattice_spacing() ** 3
    return n * (min(rho * 4.18879 * r_cut ** 3, n) - 2) / 2


def _spme_work(n, k):
    """Spreading and gathering over 125 points, four real-to-complex passes' worth of transforms, one product."""
    return n * (125 * 10 + 200) + 2 * 2.5 * k ** 3 * math.log2(k ** 3) + 2 * k ** 3


def work(case):
    """Operations of the pairs inside the cutoff (each once), of the proposals and of SPME; state read and written once a step."""
    kind = case["kind"]
    if kind == "batch":
        mean2 = (case["lo"] ** 2 + case["lo"] * case["hi"] + case["hi"] ** 2) / 3.0
        n = 1.5 * (case["lo"] + case["hi"]) * case["replicas"]
        return {"bytes": (case["steps"] + 1) * n * 96.0, "flops": (case["steps"] + 1) * case["replicas"] * 4.5 * mean2 * 55}
    n = 3 * (case["n_side"] ** 3 if case.get("n_side") else case["mol"])
    rc = case["r_cut"]
    if kind == "run":
        steps = case["steps"]
        pairs = _pairs_in(n, rc) if rc else n * n / 2
        every = {"BOUNCE_RESPA": (1, 2), "BOUNCE_RESPA1": (2, 6)}.get(case["integ"], (1, 1))
        flops = (steps / every[0] + 1) * pairs * (50 if case["n_side"] else 30) + (steps + 1) * n * 200
        if case["coul"]:
            flops += steps * n * 100 * case["dt"] * 150
        if case["n_side"]:
            flops += (steps / every[1] + 1) * _spme_work(n, _grid(case["n_side"]))
        return {"bytes": steps * n * 96.0, "flops": flops}
    if kind == "jump":
        return {"bytes": n * (24 + 24 + 24 + 32 + 8), "flops": n * 50 * 150.0}
    if kind == "forces":
        return {"bytes": 2 * n * 96.0, "flops": 2 * (_pairs_in(n, rc) * 50 + _spme_work(n, _grid(case["n_side"])))}
    if kind == "observe":
        return {"bytes": 2 * n * 48.0, "flops": 2 * (_pairs_in(n, rc) * 40 + _spme_work(n, _grid(case["n_side"])) + _pairs_in(n, 8.0) * 15)}
    if kind == "match":
        return {"bytes": n * 4 * 24.0, "flops": _pairs_in(n, rc) * (60 + 120)}
    return {"bytes": n * 40.0, "flops": (n * n / 2 * 25 if not case["n_side"] else n * n / 2 * 12 + _pairs_in(n, rc) * 30)}


# ------------------------------------------------------- 64-bit references
def _list(q, mol, box, r):
    """All pairs i < j of different molecules closer than r (minimum image)."""
    n, out = len(q), []
    rows = max(1, (1 << 27) // n)
    for b in range(0, n, rows):
        e = min(n, b + rows)
        keep = mol[b:e, None] != mol[None, :]
        keep &= torch.arange(b, e, device=DEV)[:, None] < torch.arange(n, device=DEV)[None, :]
        if math.isfinite(r):
            r2 = torch.zeros((e - b, n), dtype=torch.float64, device=DEV)
            for c in range(3):
                d = q[b:e, c, None] - q[None, :, c]
                if box is not None:
                    d -= box[c] * (d / box[c]).round()
                r2 += d * d
            keep &= r2 < r * r
        i, j = keep.nonzero(as_tuple=True)
        out.append(torch.stack((i + b, j)))
    return torch.cat(out, 1)


def _at(q, ij, box):
    d = q[ij[0]] - q[ij[1]]
    return d if box is None else d - box * (d / box).round()


def _tables(s):
    s6 = _t(s.lj_sigma) ** 6
    return 4 * _t(s.lj_eps) * s6 * s6, 4 * _t(s.lj_eps) * s6


def _pair_sums(q, s, ij, r_cut, beta):
    """Coulomb and LJ energies and the gradient over the pairs ij within r_cut."""
    box = None if s.box is None else _t(s.box)
    ty, ch = _t(s.type, torch.int64), _t(s.charge)
    d = _at(q, ij, box)
    r2 = (d * d).sum(1)
    if math.isfinite(r_cut):
        inside = r2 < r_cut * r_cut
        ij, d, r2 = ij[:, inside], d[inside], r2[inside]
    t12, t6 = _tables(s)
    i, j = ij
    wc, wl, g = _pair(r2, KCOUL * ch[i] * ch[j], t12[ty[i], ty[j]], t6[ty[i], ty[j]], beta)
    f = g[:, None] * d
    return wc.sum(), wl.sum(), torch.zeros_like(q).index_add_(0, i, f).index_add_(0, j, f, alpha=-1.0)


def _spline(fr, n):
    """M_n(fr + t) and its derivative, t = 0 .. n - 1."""
    a = [fr, 1.0 - fr] + [torch.zeros_like(fr)] * (n - 1)
    dw = None
    for k in range(2, n):
        if k == n - 1:
            dw = [a[t] - (a[t - 1] if t else 0.0) for t in range(n)]
        a = [((fr + t) * a[t] + ((k + 1 - fr - t) * a[t - 1] if t else 0.0)) / k for t in range(n + 1)]
    return torch.stack(a[:n], -1), torch.stack(dw, -1)


def _bmod(k, n):
    w = _spline(torch.zeros(1, dtype=torch.float64), n)[0][0].numpy()     # M_n(0), M_n(1), ..
    m = np.arange(k)
    s = np.abs(sum(w[t + 1] * np.exp(2j * np.pi * m * t / k) for t in range(n - 1))) ** 2
    out = np.where(s > 1e-7, 1.0 / np.maximum(s, 1e-300), 0.0)
    for i in np.nonzero(s <= 1e-7)[0]:
        out[i] = 0.5 * (1.0 / s[i - 1] + 1.0 / s[(i + 1) % k])
    return out


def _spme(q, s, k, n=5, beta=BETA):
    """Smooth particle-mesh Ewald: reciprocal, self and same-molecule energy, and the gradient."""
    box, ch = _t(s.box), _t(s.charge)
    f = q / box
    u = (f - f.floor()) * k
    fl = u.floor()
    w, dw = _spline(u - fl, n)                                             # [atoms, 3, n]
    ig = (fl.long()[:, :, None] - torch.arange(n, device=DEV)) % k
    cell = ((ig[:, 0, :, None, None] * k + ig[:, 1, None, :, None]) * k + ig[:, 2, None, None, :]).reshape(len(q), -1)

    def mix(a, b, c):
        return (a[:, :, None, None] * b[:, None, :, None] * c[:, None, None, :]).reshape(len(q), -1)

    grid = torch.zeros(k ** 3, dtype=torch.float64, device=DEV)
    grid.index_add_(0, cell.reshape(-1), (ch[:, None] * mix(w[:, 0], w[:, 1], w[:, 2])).reshape(-1))
    m = np.fft.fftfreq(k, 1.0 / k)
    m2 = [_t((m / float(s.box[c])) ** 2) for c in range(3)]
    m2 = m2[0][:, None, None] + m2[1][None, :, None] + m2[2][None, None, :]
    b = _t(_bmod(k, n))
    bc = b[:, None, None] * b[None, :, None] * b[None, None, :] * torch.exp(-math.pi ** 2 * m2 / beta ** 2) / (math.pi * float(np.prod(s.box)) * m2)
    bc[0, 0, 0] = 0.0
    ft = torch.fft.fftn(grid.reshape(k, k, k))
    energy = 0.5 * KCOUL * (bc * (ft.real ** 2 + ft.imag ** 2)).sum()
    at = (torch.fft.ifftn(ft * bc).real * k ** 3).reshape(-1)[cell]
    g = torch.stack([(at * mix(*[(dw if c == d else w)[:, c] for c in range(3)])).sum(1) * (k / box[d]) for d in range(3)], 1)
    g = KCOUL * ch[:, None] * g
    energy = energy - KCOUL * beta / math.sqrt(math.pi) * (ch * ch).sum()
    o = torch.arange(0, len(q), 3, device=DEV)
    for a, c in ((0, 1), (0, 2), (1, 2)):                                  # the pairs of one molecule
        i, j = o + a, o + c
        d = q[i] - q[j]
        r2 = (d * d).sum(1)
        r = r2.sqrt()
        qq = KCOUL * ch[i] * ch[j]
        e = torch.erf(beta * r) / r
        energy = energy - (qq * e).sum()
        h = (-qq * (2 * beta / math.sqrt(math.pi) * torch.exp(-beta ** 2 * r2) - e) / r2)[:, None] * d
        g.index_add_(0, i, h).index_add_(0, j, h, alpha=-1.0)
    return energy, g


def _match_params(requires_grad=False):
    sig, eps = torch.zeros(2, 2, dtype=torch.float64), torch.zeros(2, 2, dtype=torch.float64)
    sig[0, 0], eps[0, 0] = 3.15, 0.152
    return [t.requires_grad_(requires_grad) for t in (torch.tensor([-0.834, 0.417], dtype=torch.float64), sig, eps)]


def _match_forces(q, s, ij, qt, sig, eps):
    """Pair forces and energy as functions of positions and per-type parameters (differentiable)."""
    ty = _t(s.type, torch.int64)
    d = _at(q, ij, _t(s.box))
    r2 = (d * d).sum(1)
    ti, tj = ty[ij[0]], ty[ij[1]]
    s6 = (sig[ti, tj]) ** 6
    e4 = 4.0 * eps[ti, tj]
    wc, wl, g = _pair(r2, KCOUL * qt[ti] * qt[tj], e4 * s6 * s6, e4 * s6, BETA)
    f = g[:, None] * d
    return torch.zeros_like(q).index_add(0, ij[0], -f).index_add(0, ij[1], f), (wc + wl).sum()


def _match_target(s, r_cut):
    """Forces of the parameters to be found: sigma + 2 %, epsilon - 5 %, charges x 0.98."""
    q = _t(s.q)
    ij = _list(q, _t(s.molecule, torch.int64), _t(s.box), r_cut)
    qt, sig, eps = [p.to(DEV) for p in _match_params()]
    return _match_forces(q, s, ij, 0.98 * qt, 1.02 * sig, 0.95 * eps)[0]


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) over arrays of counters."""
    c = [np.asarray(x, dtype=np.uint64) + np.zeros_like(np.asarray(c1, dtype=np.uint64)) for x in (c0, c1, c2, c3)]
    low = np.uint64(0xFFFFFFFF)
    for r in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF), b & low,
             (a >> np.uint64(32)) ^ c[3] ^ np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF), a & low]
    return c


def _baoab(case, s, seed):
    """The BAOAB trajectory of a box or droplet: positions and velocities after the case's steps."""
    q, v, mol = _t(s.q), _t(s.v), _t(s.molecule, torch.int64)
    box = None if s.box is None else _t(s.box)
    r_cut, beta = (case["r_cut"], BETA) if case["n_side"] else (case["r_cut"] or math.inf, 0.0)
    im = ACCEL / _t(s.mass)[:, None]
    dt = case["dt"]
    c1 = math.exp(-0.001 * dt)
    sd = ((1.0 - c1 * c1) * KB * 300.0 * im).sqrt()
    ij = ref = None

    def grad():
        nonlocal ij, ref
        if ij is None or (math.isfinite(r_cut) and float((q - ref).norm(dim=1).max()) > 0.5):
            ij, ref = _list(q, mol, box, r_cut + 1.0), q.clone()
        g = _pair_sums(q, s, ij, r_cut, beta)[2] + _bonded(q, s)[2]
        return g + _spme(q, s, _grid(case["n_side"]))[1] if case["n_side"] else g

    g = grad()
    for k in range(case["steps"]):
        v = v - 0.5 * dt * im * g
        q = q + 0.5 * dt * v
        x = _philox(0, np.arange(len(q)), k, 0, 7, 0)
        u = [(a >> np.uint64(8)).astype(np.float64) * 2.0 ** -24 for a in x]
        ra, rb = np.sqrt(-2.0 * np.log(u[0] + 2.0 ** -24)), np.sqrt(-2.0 * np.log(u[2] + 2.0 ** -24))
        z = np.stack((ra * np.cos(2 * np.pi * u[1]), ra * np.sin(2 * np.pi * u[1]), rb * np.cos(2 * np.pi * u[3])), 1)
        v = c1 * v + sd * _t(z)
        q = q + 0.5 * dt * v
        g = grad()
        v = v - 0.5 * dt * im * g
    return q, v


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "jump") or (kind == "run" and case["integ"] != "BAOAB"):
        return None             # sequential chains of accepted and rejected proposals, one at a time for every atom
    s = _system(case, seed)
    if kind == "run":
        q, v = _baoab(case, s, seed)
        return {"q": q, "v": v}
    mol, box = _t(s.molecule, torch.int64), None if s.box is None else _t(s.box)
    if kind == "energy":
        r_cut, beta = (case["r_cut"], BETA) if case["n_side"] else (math.inf, 0.0)
        wc, wl, _ = _pair_sums(_t(s.q), s, _list(_t(s.q), mol, box, r_cut), r_cut, beta)
        return torch.stack((wc, wl))
    if kind == "match":
        q, p = _t(s.q).requires_grad_(True), [x.detach().to(DEV).requires_grad_(True) for x in _match_params()]
        ij = _list(q.detach(), mol, box, case["r_cut"])
        f, e = _match_forces(q, s, ij, *p)
        loss = ((f - _match_target(s, case["r_cut"])) ** 2).sum()
        return {"forces": f.detach(), "energy": e.detach(), "loss": loss.detach(), "grads": list(torch.autograd.grad(loss, [q, *p]))}
    out = []
    shift = np.random.default_rng(seed + 5).uniform(3.0, 9.0, 3)
    for q in (_t(s.q), _t(s.q + shift)):
        wc, wl, g = _pair_sums(q, s, _list(q, mol, box, case["r_cut"]), case["r_cut"], BETA)
        eb, ea, gb = _bonded(q, s)
        er, gr = _spme(q, s, _grid(case["n_side"]))
        if kind == "forces":
            out += [g + gb, gr]
        else:
            ek = (0.5 * _t(s.mass) / ACCEL * (_t(s.v) ** 2).sum(1)).sum()
            out += [{"coulomb": wc, "lj": wl, "bond": eb, "angle": ea, "kinetic": ek, "recip": er,
                     "potential": wc + wl + eb + ea + er}, None]
    return out
