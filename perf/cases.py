"""The work that a user of this framework has it do, as cases that can be timed.

A case is one call sequence through the public entry points: Langevin steps of
one or many lambda windows (solvent and complex legs, real-space or PME
electrostatics, with and without replica exchange), forces and energies of a
frame, reduced-potential rows of stored frames, the allocation-free frame call
and MBAR. Sizes are those of abfe_synth's workloads, the tests and bench.py:
672 atoms to some millions, cutoffs 0.9 to 1.2 nm, ligands of 20 to 90 atoms,
1 to 72 windows per context.

Every array is made from the seed: the structures are abfe_synth's seeded
lattice systems (one per size), every seed moves each atom of every window by
its own N(0, 0.002 nm) (about a bond's thermal width) and draws its own
Maxwell velocities. FP32 contexts (the default precision) return what they
compute as the binary32 numbers that their arithmetic and coordinates are;
FP64 contexts, the frame call, MBAR and the states return as they come.
"""
import functools
import math

import numpy as np
import torch

import abfe_synth as S
import paper_2603_22274_gb300 as G
from paper_2603_22274_gb300 import _binding as B


# --------------------------------------------------------------------- the cases

def _md(**kw):
    d = dict(kind="md", leg="complex", atoms=25000, windows=1, lig=40, cutoff=1.0, steps=50,
             graph=0, skin=0.0, prune=0.0, precision=0, pme=0, mode=0, charge=0.0, every=0)
    d.update(kw)
    return d


def _frame(**kw):
    d = dict(kind="frame", leg="solvent", atoms=4500, windows=1, lig=60, cutoff=1.0, precision=0,
             pme=0, mode=0, charge=0.0)
    d.update(kw)
    return d


def listed():
    return [
        # the smallest call: forces, energies and dU/dlambda of the 672-atom box at its 12
        # states in FP64 pair arithmetic (the framework's own smoke check); latency counts
        _frame(name="frame-tiny-f64", leg="tiny", atoms=672, windows=12, lig=24, cutoff=0.9,
               precision=1),
        # one solvent-leg window of a charged ligand (alchemical waters): a host program asks
        # for device forces, energies and dU/dlambda at the current coordinates
        _frame(name="frame-solvent-charged", charge=1.0),
        # one frame of several complex windows with the paper's full PME electrostatics
        _frame(name="frame-pme", leg="complex", atoms=25000, windows=4, lig=20, cutoff=0.9, pme=4),
        # stored frames of a complex leg are re-evaluated: set_positions, then the u_kn rows at
        # all 24 states (list build, prune, energy pass and state sums in one call chain)
        dict(_frame(name="ukn-frames", leg="complex", atoms=25000, windows=8, lig=20, cutoff=0.9),
             kind="ukn"),
        # one solvent-leg window stepped alone in a captured loop: launches and gaps count
        _md(name="md-solvent", leg="solvent", atoms=4500, lig=60, steps=100, graph=50, skin=0.2,
            prune=0.06),
        # one 60,000-atom complex window as a user gets it without tuning: direct launches
        _md(name="md-complex", atoms=60000, lig=60, steps=60),
        # 24 windows of a 25,000-atom complex, tuned, graph-captured
        _md(name="md-loop", windows=24, lig=20, cutoff=0.9, steps=50, graph=50, skin=0.25,
            prune=0.1),
        # a ligand's whole path in one context: 42 complex windows of 40,000 atoms and 30
        # solvent windows of 4,500 (uneven windows in one launch); the largest
        _md(name="md-batch", leg="both", atoms=40000, windows=72, lig=60, steps=40, graph=40,
            skin=0.3, prune=0.1),
        # windows with PME on every step
        _md(name="md-pme", windows=8, lig=20, cutoff=0.9, steps=30, graph=30, skin=0.25, prune=0.1,
            pme=4),
        # 12 windows of a small complex with an in-loop replica exchange every 10 steps
        _md(name="md-exchange", atoms=6000, windows=12, lig=30, steps=40, graph=20, skin=0.2,
            prune=0.06, every=10),
        # the frame call of a host MD engine's plugin: one 60,000-atom frame at 42 states
        dict(name="noalloc-complex", kind="noalloc", leg="complex", atoms=60000, lig=60, cutoff=1.0,
             mode=0),
        # MBAR of one 80-window segment, 2,000 samples a window, u_kn resident on the device
        dict(name="mbar-80", kind="mbar", states=80, samples=2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    cutoff = rng.choice([0.9, 1.0, 1.0, 1.1, 1.2])
    lig = rng.randint(20, 90)
    kind = rng.choice(["md", "md", "md", "md", "frame", "frame", "ukn", "noalloc", "mbar"])
    leg = rng.choice(["solvent", "complex", "complex"])
    mode = rng.choice([0, 0, 0, 1])
    if kind == "mbar":
        states = _log(rng, 5, 128)
        return dict(kind=kind, states=states, samples=_log(rng, 200, min(4000, 160000 // states + 200)))
    if kind == "noalloc":
        return dict(kind=kind, leg=leg, lig=lig, cutoff=cutoff, mode=mode,
                    atoms=_log(rng, 6000, 100000) if leg == "complex" else _log(rng, 3300, 9000))
    # (even B-spline orders: the moduli of odd orders are singular on even grids)
    pme = rng.choice([0, 0, 0, 4, 4, 6]) if mode == 0 else 0
    charge = rng.choice([0.0, 0.0, 1.0, -1.0]) if pme == 0 else 0.0
    atoms = _log(rng, 6000, 60000) if leg == "complex" else _log(rng, 3300, 9000)
    if kind != "md":
        most = max(1, 200000 // atoms)
        return dict(_frame(leg=leg, atoms=atoms, windows=min(12, _log(rng, 1, most)), lig=lig,
                           cutoff=cutoff, pme=pme if kind == "frame" else 0, mode=mode, charge=charge,
                           precision=1 if kind == "frame" and atoms < 5000 and rng.random() < 0.5 else 0),
                    kind=kind)
    windows = min(30, _log(rng, 1, max(1, 900000 // atoms)))
    steps = max(5, min(_log(rng, 10, 100), 25000000 // (atoms * windows)))
    skin = rng.choice([0.15, 0.2, 0.25, 0.3])
    tuned = rng.random() < 0.7
    return _md(leg=leg, atoms=atoms, windows=windows, lig=lig, cutoff=cutoff, steps=steps, mode=mode,
               pme=pme, charge=charge, graph=steps if tuned else 0, skin=skin if tuned else 0.0,
               prune=rng.choice([0.04, 0.06, 0.1]) if tuned else 0.0,
               every=10 if 1 < windows <= 24 and rng.random() < 0.25 else 0)


# --------------------------------------------------------------------- the inputs

@functools.lru_cache(maxsize=32)
def _system(leg, atoms, lig, charge):
    if leg == "tiny":
        return S.tiny()
    for k in range(20):   # another chain where this one does not fit beside the core
        ligand = S.make_ligand(np.random.default_rng(1234 + lig + 1000 * k), lig)
        try:
            if leg == "solvent":
                s = S.solvent_leg(1235 + atoms, ligand=ligand, box=(atoms / 105.0) ** (1 / 3),
                                  n_atoms=atoms)
            else:
                s = S.complex_leg(1236 + atoms, n_atoms=atoms, ligand=ligand,
                                  core_diameter=min(4.5, 0.55 * (atoms / 100.0) ** (1 / 3)))
        except RuntimeError:
            continue
        return S.charged_leg(s, charge) if charge else s
    raise RuntimeError("no ligand could be placed")


def _schedule(leg, cutoff):
    if leg == "tiny":
        return S.schedule_k12()
    if leg == "solvent":
        return S.schedule_solvent_k30()
    return S.schedule_k24() if cutoff == 0.9 else S.schedule_k42()


def _windows(c):
    """(systems, system of each window, schedules, schedule and state of each window)."""
    q = c.get("charge", 0.0)
    if c["leg"] == "both":
        systems = [_system("complex", c["atoms"], c["lig"], q), _system("solvent", 4500, c["lig"], q)]
        scheds = [S.schedule_k42(), S.schedule_solvent_k30()]
        n = c["windows"] * 42 // 72
        of = [0] * n + [1] * (c["windows"] - n)
        st = [k % 42 for k in range(n)] + [k % 30 for k in range(c["windows"] - n)]
        return systems, of, scheds, of, st
    sch = _schedule(c["leg"], c["cutoff"])
    R = c.get("windows", 1)
    st = [(k * sch.K) // R for k in range(R)] if R > 1 else [sch.K // 2]
    return [_system(c["leg"], c["atoms"], c["lig"], q)], [0] * R, [sch], [0] * R, st


def _params(c):
    p = S.params_for(c["cutoff"], round(3.12 / c["cutoff"], 2), ligand_mode=c.get("mode", 0))
    if c["leg"] == "tiny":
        p["skin"] = 0.0
    if c.get("pme", 0):
        p.update(pme_order=c["pme"], pme_spacing=0.12)
    return p


def _frames(c, seed):
    """Positions and velocities of every window, binary32-representable, in the box."""
    systems, of, _, _, _ = _windows(c)
    rng = np.random.default_rng(seed)
    kT = _params(c)["kT"]
    X, V = [], []
    for s in of:
        t = systems[s]
        box = t.box.astype(np.float32)
        x = t.pos.astype(np.float32) + np.float32(0.002) * rng.standard_normal((t.n, 3), np.float32)
        x = np.mod(x, box)
        X.append(np.where(x >= box, np.float32(0), x))
        V.append(rng.standard_normal((t.n, 3), np.float32) * np.sqrt(kT / t.mass)[:, None].astype(np.float32))
    return np.concatenate(X).astype(np.float64), np.concatenate(V).astype(np.float64)


def _mbar_inputs(c, seed):
    """u_kn of harmonic states whose stiffness grows by 1.25 a window (neighbours overlap as an
    alchemical schedule's do), with uneven sample counts."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = 1.25 ** torch.arange(c["states"], dtype=torch.float64, device="cuda")
    n_k = [c["samples"] + (7 * i) % 11 - 5 for i in range(c["states"])]
    of = torch.repeat_interleave(torch.arange(c["states"], device="cuda"),
                                 torch.tensor(n_k, device="cuda"))
    x = torch.randn(len(of), generator=g, dtype=torch.float64, device="cuda") / k[of].sqrt()
    return 0.5 * k[:, None] * (x * x)[None, :], np.array(n_k, np.int32)


def _noalloc_frame(c, s, p, sch, x):
    dev = "cuda"
    f = B.NoallocFrame()
    f.n_atoms = s.n
    f.box[:] = [float(v) for v in s.box]
    lig = np.where(s.is_ligand)[0].astype(np.int32)
    excl = np.full((len(lig), B.NOALLOC_MAX_EXCL), -1, np.int32)
    for r, a in enumerate(lig):
        e = np.asarray(s.excl)
        e = np.concatenate([e[e[:, 0] == a, 1], e[e[:, 1] == a, 0]])
        excl[r, :len(e)] = e
    t = [torch.tensor(np.asarray(v), dtype=d, device=dev)
         for v, d in ((x, torch.float32), (s.charge, torch.float32), (s.sigma, torch.float32),
                      (s.epsilon, torch.float32), (s.is_ligand, torch.uint8), (lig, torch.int32),
                      (excl, torch.int32))]
    f.pos, f.charge, f.sigma, f.epsilon, f.is_ligand, f.lig_idx, f.lig_excl = [v.data_ptr() for v in t]
    f.n_lig, f.K = len(lig), sch.K
    f.lam_r[:sch.K], f.lam_q[:sch.K], f.lam_v[:sch.K] = list(sch.lam_r), list(sch.lam_q), list(sch.lam_v)
    f.cutoff, f.ewald_beta, f.sc_alpha, f.sc_p = p["cutoff"], p["ewald_beta"], p["sc_alpha"], p["sc_p"]
    f.coulomb_k, f.ligand_mode = p["coulomb_k"], p["ligand_mode"]
    b = s.boresch
    if b is not None:
        f.has_boresch = 1
        f.anchors[:] = [int(v) for v in b.anchors]
        f.b_r0, f.b_kr, f.b_ktheta, f.b_kphi = b.r0, b.k_r, b.k_theta, b.k_phi
        f.b_theta0[:] = [float(v) for v in b.theta0]
        f.b_phi0[:] = [float(v) for v in b.phi0]
    return f, t


def prepare(case, seed):
    c = case
    if c["kind"] == "mbar":
        u, n_k = _mbar_inputs(c, seed)
        return dict(case=c, u=u, n_k=n_k)
    systems, of, scheds, sched_of, state = _windows(c)
    p = _params(c)
    if c["kind"] == "noalloc":
        x, _ = _frames(c, seed)
        f, keep = _noalloc_frame(c, systems[0], p, scheds[0], x)
        return dict(case=c, frame=f, keep=keep,
                    du=torch.zeros(f.K, dtype=torch.float64, device="cuda"))
    w = S.Workload("case", systems, np.array(of, np.int32), scheds, np.array(sched_of, np.int32),
                   np.array(state, np.int32), p)
    x, v = _frames(c, seed)
    stream = torch.cuda.Stream()
    e = G.engine_for_workload(w, stream=stream, precision=c["precision"])
    st = dict(case=c, engine=e, stream=stream)
    if c["kind"] == "ukn":
        return dict(st, x=x)
    e.set_positions(x)
    if c["kind"] == "md":
        e.set_velocities(v)
        if c["skin"]:
            e.set_tuning(group=1, max_entries=512, block_threads=256, graph_steps=c["graph"],
                         skin=c["skin"], prune_skin=c["prune"])
        if c["every"]:
            e.set_exchange(c["every"], seed=seed)
        return dict(st, seed=seed)
    if c["precision"] == 0:
        st.update(f=torch.zeros(e.total_atoms, 3, device="cuda"),
                  e=torch.zeros(e.R, G.N_ENERGY, dtype=torch.float64, device="cuda"),
                  d=torch.zeros(e.R, G.N_DUDL, dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    if c["kind"] == "mbar":
        f, _ = G.mbar(state["u"], state["n_k"], tol=1e-10)
        return f
    if c["kind"] == "noalloc":
        import ctypes
        st = G.lib().abfe_ukn_frame_noalloc(ctypes.byref(state["frame"]), state["du"].data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        if st != 0:
            raise RuntimeError(f"abfe_ukn_frame_noalloc: status {st}")
        return state["du"]
    e = state["engine"]
    if c["kind"] == "md":
        # the sampling loop: n steps, then the frame as a trajectory file takes it
        e.step(c["steps"], dt=0.001, gamma=5.0, seed=state["seed"])
        out = dict(pos=e.positions().astype(np.float32))
        if c["every"]:
            out["states"] = e.replica_states()
        return out
    if c["kind"] == "ukn":
        e.set_positions(state["x"])
        return dict(zip(("ukn", "du", "dudl"), (a.astype(np.float32) for a in e.eval_ukn())))
    if c["precision"] == 1:
        return dict(zip(("forces", "energy", "dudl"), e.compute()))
    e.compute_device(state["f"], state["e"], state["d"])
    with torch.cuda.stream(state["stream"]):
        return dict(forces=state["f"], energy=state["e"].float(), dudl=state["d"].float())


def work(case):
    """Inputs and outputs once (position, velocity, parameters in; position, velocity or force
    out) and 61 flops per in-cutoff pair and step (the pair terms of plain LJ and erfc Coulomb
    and both force accumulations, FMA = 2), 12 per ligand pair and state. MBAR: one application
    of its map (two multiply-adds a matrix element)."""
    c = case
    if c["kind"] == "mbar":
        el = c["states"] * c["states"] * c["samples"]
        return dict(bytes=8 * el, flops=4 * el)
    systems, of, scheds, sched_of, _ = _windows(c)
    n = pairs = lig_pairs = states = 0.0
    for s, h in zip(of, sched_of):
        t = systems[s]
        near = t.n / float(np.prod(t.box)) * 4.0 / 3.0 * math.pi * c["cutoff"] ** 3
        n += t.n
        pairs += 0.5 * t.n * near
        lig_pairs += t.n_ligand * near * len(set(scheds[h].lam_v))
        states += scheds[h].K
    if c["kind"] == "noalloc":
        return dict(bytes=25 * n + 8 * states, flops=12 * lig_pairs + 8 * n)
    if c["kind"] == "md":
        return dict(bytes=64 * n, flops=c["steps"] * (61 * pairs + 60 * n))
    if c["kind"] == "ukn":
        return dict(bytes=40 * n + 16 * states, flops=61 * pairs + 12 * lig_pairs)
    return dict(bytes=40 * n, flops=61 * pairs)


# --------------------------------------------------------------------- 64-bit values

def _near_image(d, box):
    return d - box * torch.round(d / box)


class _Exact:
    """One window's terms at positions x, each written out from its definition, all pairs."""

    def __init__(self, s, p, x):
        t = functools.partial(torch.tensor, dtype=torch.float64, device="cuda")
        self.p, self.s = p, s
        self.x = t(x)
        self.x.requires_grad_(True)
        self.box, self.q, self.sig, self.eps = t(s.box), t(s.charge), t(s.sigma), t(s.epsilon)
        self.lig = torch.tensor(s.is_ligand.astype(bool), device="cuda")
        self.dq = torch.zeros_like(self.q)
        if len(s.alch_water):
            self.dq[torch.tensor(s.alch_water, device="cuda").long()] = t(s.alch_water_dq)
        ex = np.sort(np.asarray(s.excl, np.int64), axis=1)
        self.ex = torch.tensor(ex, device="cuda")
        key = torch.tensor(ex[:, 0] * s.n + ex[:, 1], device="cuda")
        got = []
        y = self.x.detach()
        for a in range(0, s.n, 1024):
            r2 = sum(_near_image(y[None, :, k] - y[a:a + 1024, None, k], self.box[k]) ** 2 for k in range(3))
            i, j = torch.nonzero(r2 < p["cutoff"] ** 2, as_tuple=True)
            i = i + a
            ok = j > i
            i, j = i[ok], j[ok]
            ok = ~torch.isin(i * s.n + j, key)
            got.append((i[ok], j[ok]))
        self.i, self.j = (torch.cat(v) for v in zip(*got))

    def charges(self, lq):
        q = self.q + (1.0 - lq) * self.dq
        return torch.where(self.lig, lq * q, q)

    def pairs(self, i, j, lq, lv):
        """Six sums: LJ and Coulomb of env-env, LJ of lig-env and lig-lig, Coulomb of both."""
        p = self.p
        d = _near_image(self.x[j] - self.x[i], self.box)
        r2 = (d * d).sum(1)
        r = r2.sqrt()
        n = self.lig[i].long() + self.lig[j].long()
        q = self.charges(lq)
        if p["ligand_mode"] == 1:
            full = self.q + (1.0 - lq) * self.dq
            qq = torch.where(n == 2, full[i] * full[j], q[i] * q[j])
        else:
            qq = q[i] * q[j]
        ec = p["coulomb_k"] * qq * torch.erfc(p["ewald_beta"] * r) / r
        s6 = (0.5 * (self.sig[i] + self.sig[j])) ** 6
        e4 = 4.0 * torch.sqrt(self.eps[i] * self.eps[j])
        r6 = r2 * r2 * r2
        soft = (n == 1) | ((n == 2) & (p["ligand_mode"] == 0))
        A = torch.where(soft, p["sc_alpha"] * (1.0 - lv) ** p["sc_p"], torch.zeros_like(r))
        a = s6 / (A * s6 + r6)
        el = torch.where(soft, lv, torch.ones_like(lv)) * e4 * (a * a - a)
        return [el[n == 0].sum(), ec[n == 0].sum(), el[n == 1].sum(), el[n == 2].sum(),
                ec[n == 1].sum(), ec[n == 2].sum()]

    def bonds(self):
        s = self.s
        t = functools.partial(torch.tensor, dtype=torch.float64, device="cuda")
        b = torch.tensor(s.bonds, device="cuda").long()
        d = _near_image(self.x[b[:, 1]] - self.x[b[:, 0]], self.box)
        return (0.5 * t(s.bond_k) * (d.norm(dim=1) - t(s.bond_r0)) ** 2).sum()

    def dihedral(self, a, b, c, d):
        b1, b2, b3 = (_near_image(self.x[v] - self.x[u], self.box) for u, v in ((a, b), (b, c), (c, d)))
        n1, n2 = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
        return torch.atan2(b2.norm(dim=-1) * (b1 * n2).sum(-1), (n1 * n2).sum(-1))

    def torsions(self):
        s = self.s
        if not len(s.torsions):
            return self.x.sum() * 0.0
        t = functools.partial(torch.tensor, dtype=torch.float64, device="cuda")
        phi = self.dihedral(*torch.tensor(s.torsions, device="cuda").long().T)
        return (t(s.torsion_k) * (1.0 + torch.cos(t(s.torsion_n) * phi - t(s.torsion_phi0)))).sum()

    def restraint(self):
        b = self.s.boresch
        if b is None:
            return self.x.sum() * 0.0
        P1, P2, P3, L1, L2, L3 = (int(a) for a in b.anchors)
        sep = lambda u, v: _near_image(self.x[v] - self.x[u], self.box)  # noqa: E731
        U = 0.5 * b.k_r * (sep(P1, L1).norm() - b.r0) ** 2
        for (u, v, w), t0 in zip(((P1, L1, L2), (L1, P1, P2)), b.theta0):
            m, n = sep(v, u), sep(v, w)
            U = U + 0.5 * b.k_theta * (torch.acos((m * n).sum() / (m.norm() * n.norm())) - float(t0)) ** 2
        for q, f0 in zip(((P2, P1, L1, L2), (P1, L1, L2, L3), (L1, P1, P2, P3)), b.phi0):
            U = U + b.k_phi * (1.0 - torch.cos(self.dihedral(*q) - float(f0)))
        return U

    def reciprocal(self, lq):
        """Smooth PME at the order and spacing of the case, the self term, excluded pairs."""
        p = self.p
        if not p.get("pme_order", 0):
            return self.x.sum() * 0.0
        po, beta, ke = p["pme_order"], p["ewald_beta"], p["coulomb_k"]
        L = [float(v) for v in self.s.box]

        def good(n):
            for f in (2, 3, 5):
                while n % f == 0:
                    n //= f
            return n == 1

        K = [next(n for n in range(max(2 * po, math.ceil(v / p["pme_spacing"] - 1e-9)), 1000) if good(n))
             for v in L]

        def spline(n, u):
            if n == 2:
                return torch.clamp(1.0 - (u - 1.0).abs(), min=0.0)
            return (u * spline(n - 1, u) + (n - u) * spline(n - 1, u - 1.0)) / (n - 1)

        q = self.charges(lq)
        idx, w = [], []
        for a in range(3):
            u = self.x[:, a] / L[a] * K[a]
            base = torch.floor(u.detach())
            k = base[:, None] - torch.arange(po, device="cuda")
            idx.append(torch.remainder(k, K[a]).long())
            w.append(spline(po, u[:, None] - k))
        at = (idx[0][:, :, None, None] * K[1] + idx[1][:, None, :, None]) * K[2] + idx[2][:, None, None, :]
        val = q[:, None, None, None] * w[0][:, :, None, None] * w[1][:, None, :, None] * w[2][:, None, None, :]
        Q = torch.zeros(K[0] * K[1] * K[2], dtype=torch.float64, device="cuda")
        Q = Q.index_add(0, at.reshape(-1), val.reshape(-1)).reshape(K)
        m2, bb = 0.0, 1.0
        for a in range(3):
            f = torch.fft.fftfreq(K[a], 1.0 / K[a], dtype=torch.float64, device="cuda")
            m2 = m2 + ((f / L[a]) ** 2).reshape([-1 if a == k else 1 for k in range(3)])
            t = torch.arange(po - 1, device="cuda", dtype=torch.float64)
            ang = 2.0 * math.pi * f[:, None] * t[None, :] / K[a]
            M = spline(po, t + 1.0)
            den = (M * torch.cos(ang)).sum(1) ** 2 + (M * torch.sin(ang)).sum(1) ** 2
            bb = bb * (1.0 / den).reshape([-1 if a == k else 1 for k in range(3)])
        C = torch.exp(-(math.pi / beta) ** 2 * m2) / (math.pi * L[0] * L[1] * L[2] * m2)
        C[0, 0, 0] = 0.0
        E = 0.5 * ke * (bb * C * torch.fft.fftn(Q).abs() ** 2).sum()
        E = E - ke * beta / math.sqrt(math.pi) * (q * q).sum()
        i, j = self.ex[:, 0], self.ex[:, 1]
        r = _near_image(self.x[j] - self.x[i], self.box).norm(dim=1)
        return E - ke * (q[i] * q[j] * torch.erf(beta * r) / r).sum()

    def all_terms(self, lam):
        """Energy components in the order of ENERGY_NAMES (the last their sum), forces, dU/dlambda."""
        l3 = [torch.tensor(float(v), dtype=torch.float64, device="cuda", requires_grad=True) for v in lam]
        lr, lq, lv = l3
        ut = self.torsions()
        E = self.pairs(self.i, self.j, lq, lv) + [
            self.bonds(), lr * self.restraint(), self.reciprocal(lq),
            lv * ut if self.p["ligand_mode"] == 0 else ut]
        U = sum(E)
        g = torch.autograd.grad(U, [self.x] + l3, allow_unused=True)
        D = [torch.zeros((), dtype=torch.float64, device="cuda") if v is None else v for v in g[1:]]
        return torch.stack(E + [U]).detach(), -g[0], torch.stack(D).detach()

    def rows(self, sch, k_own):
        """U_k - U_indep at every state, U_indep, dU/dlambda at the own state."""
        dep = self.lig[self.i] | self.lig[self.j] | (self.dq[self.i] != 0) | (self.dq[self.j] != 0)
        i, j = self.i[dep], self.j[dep]
        one = torch.ones((), dtype=torch.float64, device="cuda")
        E, _, D = self.all_terms(sch.state(k_own))
        with torch.no_grad():
            base = self.pairs(i, j, one, one)
            rest = self.pairs(self.i[~dep], self.j[~dep], one, one)
            ut, ub = self.torsions(), self.restraint()
            ann = self.p["ligand_mode"] == 0
            inner = 0.0 if ann else base[3] + base[5] + ut
            du = []
            for k in range(sch.K):
                lr, lq, lv = sch.state(k)
                U = sum(self.pairs(i, j, lq * one, lv * one)) + lr * ub + (lv * ut if ann else ut)
                du.append(U - base[0] - base[1] - inner)
            indep = rest[0] + rest[1] + base[0] + base[1] + inner + self.bonds()
        return torch.stack(du), indep, D


def exact(case, seed):
    c = case
    if c["kind"] == "md":
        return None
    if c["kind"] == "mbar":
        u, n_k = _mbar_inputs(c, seed)
        ln = torch.log(torch.tensor(n_k, dtype=torch.float64, device="cuda"))
        f = torch.zeros(c["states"], dtype=torch.float64, device="cuda")
        for _ in range(20000):
            ld = torch.logsumexp((ln + f)[:, None] - u, 0)
            new = -torch.logsumexp(-u - ld, 1)
            new = new - new[0]
            d = (new - f).abs().max()
            f = new
            if d < 1e-10:
                break
        return f
    systems, of, scheds, sched_of, state = _windows(c)
    if sum(float(systems[s].n) ** 2 for s in of) > 2.5e10:
        return None
    p = _params(c)
    x, _ = _frames(c, seed)
    if c["kind"] == "noalloc":
        s, sch = systems[0], scheds[0]
        t = _Exact(s, p, x)
        dep = (t.lig[t.i] | t.lig[t.j]) & ~(t.lig[t.i] & t.lig[t.j] & (p["ligand_mode"] == 1))
        with torch.no_grad():
            ub = t.restraint()
            one = torch.ones((), dtype=torch.float64, device="cuda")
            return torch.stack([sum(t.pairs(t.i[dep], t.j[dep], sch.lam_q[k] * one, sch.lam_v[k] * one))
                                + sch.lam_r[k] * ub for k in range(sch.K)])
    got, at = [], 0
    for s, h, k in zip(of, sched_of, state):
        t = _Exact(systems[s], p, x[at:at + systems[s].n])
        at += systems[s].n
        got.append(t.rows(scheds[h], k) if c["kind"] == "ukn" else t.all_terms(scheds[h].state(k)))
        del t
    if c["kind"] == "ukn":
        du = torch.stack([g[0] for g in got])
        return dict(ukn=(du + torch.stack([g[1] for g in got])[:, None]) / p["kT"], du=du,
                    dudl=torch.stack([g[2] for g in got]))
    return dict(forces=torch.cat([g[1] for g in got]), energy=torch.stack([g[0] for g in got]),
                dudl=torch.stack([g[2] for g in got]))
