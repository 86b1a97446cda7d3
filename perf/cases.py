"""The work that users of the lambda-ABF engine have it do, as cases to time.

Every case goes through the engine's public entry points: multiple-walker MD
(`Engine.step` with the read-outs of a production loop), the host-driven form
(`set_states`, `step`, `get_states`), single energy/force evaluations
(`energy_forces`), differentiation (`autograd.energy`) and the
allocation-free alchemical pass (`alch_pairs_static`).  Inputs are seeded
synthetic systems of the shapes in `paper_2307_08006_gb300/synth.py`: water
molecules on their lattice in random orientations, jittered, with
Maxwell-Boltzmann velocities.

`exact` restates the method in 64 bits with torch and numpy only: O(N^2)
minimum-image pairs, BAOAB, Philox normals, textbook ABF.
"""
import functools
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2307_08006_gb300 import autograd, labf, synth

DENSITY_WATERS = 32.768  # waters per nm^3 of the synthetic boxes
UNEVEN = ",".join(map(str, synth.UNEVEN_WATERS))
UNEVEN_SOLUTES = ",".join(map(str, synth.UNEVEN_SOLUTES))


def _md(kind, steps, **kw):
    """An MD case: `steps` steps, then every walker's state and the ABF
    statistics are read, as a production loop writes a frame."""
    c = dict(kind=kind, steps=steps, skin=0.15, prune=0.06, tune=1, theta=0, copies=1, drive=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest production run: 4 walkers of a 257-atom LJ fluid at
        # the default options; launches and latency count
        dict(name="lj_fluid", **_md("lj", 100, cells=4, walkers=4, skin=0.3, prune=0.0, tune=0)),
        # two-stage water with the solute-parameter statistics on (dA/dtheta),
        # default options, a step count that is no multiple of the graph's
        dict(name="water256_theta", **_md("water", 25, waters="256", solutes="4", walkers=8, skin=0.1,
                                          prune=0.0, tune=0, theta=1)),
        # lambda-mass / friction sweep: 18 small systems of 8 walkers in one
        # batch (144 walkers)
        dict(name="sweep_144", **_md("water", 20, waters="256", solutes="4", walkers=8, skin=0.1, prune=0.0,
                                     tune=0, copies=18)),
        # a user with two walkers of one mid-size box at the default options
        dict(name="two_walkers", **_md("water", 33, waters="3001", solutes="17", walkers=2, skin=0.1,
                                       prune=0.0, tune=0)),
        # the solvation workload of the benchmark: 16 walkers x 12 300 atoms
        dict(name="solvation_16", **_md("water", 20, waters="4096", solutes="12", walkers=16)),
        # the same driven by a host program that keeps the state (exchange or
        # replica moves between calls): states in, 10 steps, states out
        dict(name="solvation_hosted", **_md("water", 10, waters="4096", solutes="12", walkers=16, drive=1)),
        # eight boxes of 256 to 8192 waters, 8 walkers each, in one batch
        dict(name="uneven_64", **_md("water", 10, waters=UNEVEN, solutes=UNEVEN_SOLUTES, walkers=8)),
        # the largest: a restrained complex, 16 walkers x 96 040 atoms
        dict(name="complex_16", **_md("complex", 10, waters=31000, walkers=16)),
        # differentiation: U and its gradients by x, lambda and the solute's
        # (epsilon, sigma, q), lists rebuilt from x on every call
        dict(name="gradient", kind="gradient", waters=4096, solutes=12),
        # one energy/force evaluation read on the host (rescoring a frame)
        dict(name="forces", kind="forces", waters=8192, solutes=40),
        # the allocation-free alchemical pass: the solvation system, and the
        # largest shapes a caller with a declared footprint brings
        dict(name="static_12300", kind="static", waters=4096, solutes=12),
        dict(name="static_large", kind="static", waters=40000, solutes=200),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lj", "water", "water", "water", "batch", "hosted", "complex", "gradient", "forces", "static"])
    if kind == "lj":
        return _md("lj", log_int(20, 150), cells=rng.randint(4, 8), walkers=rng.randint(1, 16), skin=0.3, prune=0.0,
                   tune=0, theta=rng.randint(0, 1))
    if kind in ("water", "hosted"):
        tuned = rng.randint(0, 1)
        return _md("water", rng.randint(5, 35), waters=str(log_int(256, 8192)), solutes=str(log_int(4, 40)),
                   walkers=2 * rng.randint(1, 8), skin=0.15 if tuned else 0.1, prune=0.06 if tuned else 0.0,
                   tune=tuned, theta=rng.randint(0, 1), drive=int(kind == "hosted"))
    if kind == "batch":
        k = rng.randint(2, 8)
        return _md("water", rng.randint(5, 20), waters=",".join(str(log_int(256, 6000)) for _ in range(k)),
                   solutes=",".join(str(log_int(4, 40)) for _ in range(k)), walkers=2 * rng.randint(1, 4))
    if kind == "complex":
        return _md("complex", rng.randint(3, 10), waters=log_int(4000, 30000), walkers=2 * rng.randint(1, 7))
    if kind == "static":
        return dict(kind="static", waters=log_int(256, 43000), solutes=log_int(1, 250))
    return dict(kind=kind, waters=log_int(256, 8192), solutes=log_int(4, 40))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _template(kind, waters, solutes):
    """The lattice system of a size (topology and force field), made once."""
    if kind == "complex":
        return synth.large_complex(n_waters=waters, n_chain=max(64, round(waters * 3000 / 31000)))
    box = (waters / DENSITY_WATERS) ** (1.0 / 3.0)
    return synth.water_box(waters, solutes, box=box, r_cut=min(1.0, math.floor(20.0 * (box / 2.0 - 0.11)) / 20.0))


def _turned(spec, waters, rng, jitter):
    """The template with every water turned about its oxygen and every atom
    jittered."""
    x = spec.x.astype(np.float64)
    w = x[:3 * waters].reshape(waters, 3, 3)
    d = w[:, 1:] - w[:, :1]
    d -= spec.box * np.round(d / spec.box)
    q = rng.standard_normal((waters, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    s, u = q[:, :1, None], q[:, None, 1:]
    u = np.broadcast_to(u, d.shape)
    t = 2.0 * np.cross(u, d)
    w[:, 1:] = w[:, :1] + d + s * t + np.cross(u, t)
    x = (x + rng.uniform(-jitter, jitter, x.shape)) % spec.box
    return replace(spec, x=x.astype(np.float32))


def _systems(case, seed):
    """[(spec, run, state)] of an MD case."""
    out = []
    if case["kind"] == "lj":
        spec = synth.lj_fluid(seed=seed % (1 << 31), cells=case["cells"])
        run = replace(synth.lj_fluid_run(seed=seed % (1 << 31), n_walkers=case["walkers"]), skin=case["skin"],
                      theta_stats=bool(case["theta"]))
        lam0 = [(k + 0.5) / case["walkers"] for k in range(case["walkers"])]
        return [(spec, run, synth.initial_state(spec, run, lam0=lam0))]
    if case["kind"] == "complex":
        sizes = [(case["waters"], 0)]
    else:
        sizes = list(zip(map(int, case["waters"].split(",")), map(int, case["solutes"].split(","))))
    for k in range(case["copies"]):
        for n_waters, n_solute in sizes:
            sd = (seed + 7919 * len(out)) % (1 << 31)
            rng = np.random.default_rng(sd)
            spec = _turned(_template(case["kind"], n_waters, n_solute), n_waters, rng,
                           0.005 if case["kind"] == "complex" else 0.01)
            # a box that is too small for the wider list keeps the default skin
            skin = case["skin"] if spec.box >= 2.0 * (spec.r_cut + case["skin"]) else 0.1
            per_stage = case["walkers"] // 2
            run = replace(synth.water_run(seed=sd, walkers_per_stage=per_stage, skin=skin),
                          theta_stats=bool(case["theta"]), m_lambda=synth.M_LAMBDA_KJ_PS2 * 10.0 ** (k % 3 - 1))
            lam0 = [0.5 * (q + 0.5) / per_stage + h for h in (0.0, 0.5) for q in range(per_stage)]
            out.append((spec, run, synth.initial_state(spec, run, lam0=lam0)))
    return out


def _one_walker(case, seed):
    """(spec, run, state) of a single evaluation on a water box."""
    rng = np.random.default_rng(seed)
    spec = _turned(_template("water", case["waters"], case["solutes"]), case["waters"], rng, 0.01)
    run = replace(synth.fixed_lambda_windows(synth.water_run(seed=seed % (1 << 31), walkers_per_stage=1), 1)[0],
                  stages=[synth.Stage(0.0, 1.0, 1, 1)])
    return spec, run, synth.initial_state(spec, run, lam0=[float(rng.uniform(0.05, 0.95))])


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    if case["kind"] in ("lj", "water", "complex"):
        systems = _systems(case, seed)
        options = dict(autotune=case["tune"], prune_margin=case["prune"])
        eng = labf.Engine([labf.SystemInput(*s) for s in systems], options=options)
        rows = int(eng.walker_rows[-1])
        x, v = (torch.empty((rows, 3), dtype=torch.float32, pin_memory=True).numpy() for _ in range(2))
        st = dict(case=case, eng=eng, x=x, v=v, stages=[(i, k) for i, s in enumerate(systems)
                                                       for k in range(len(s[1].stages))])
        if case["drive"]:  # the program keeps its walkers' state in its own page-locked arrays
            x[:] = np.concatenate([s[2].x.reshape(-1, 3) for s in systems])
            v[:] = np.concatenate([s[2].v.reshape(-1, 3) for s in systems])
            st["lam"] = np.concatenate([s[2].lam for s in systems])
            st["plam"] = np.concatenate([s[2].plam for s in systems])
        return st
    spec, run, state = _one_walker(case, seed)
    if case["kind"] == "static":
        t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)  # noqa: E731
        f = torch.float32
        return dict(case=case, args=(t(spec.x, f), t(spec.charge, f), t(spec.sigma, f), t(spec.epsilon, f),
                                     t(spec.alch, torch.uint8), t(spec.excl_group, torch.int32),
                                     t(np.nonzero(spec.alch)[0], torch.int32), spec.box, spec.r_cut, spec.eps_rf,
                                     spec.coul, float(state.lam[0]), spec.b_v, spec.b_e),
                    forces=torch.empty((spec.n, 3), dtype=f, device=dev),
                    out=torch.empty(6, dtype=torch.float64, device=dev))
    eng = labf.Engine([labf.SystemInput(spec, run, state)])
    st = dict(case=case, eng=eng)
    if case["kind"] == "gradient":
        st["x"] = torch.as_tensor(spec.x, device=dev).requires_grad_(True)
        st["lam"] = torch.tensor(float(state.lam[0]), dtype=torch.float64, device=dev, requires_grad=True)
        st["theta"] = torch.as_tensor(autograd.theta_of(spec), device=dev).requires_grad_(True)
    return st


def run(state):
    case = state["case"]
    if case["kind"] in ("lj", "water", "complex"):
        eng = state["eng"]
        if case["drive"]:
            eng.set_states(x=state["x"], v=state["v"], lam=state["lam"], plam=state["plam"])
        eng.step(case["steps"])
        out = eng.get_states(x=state["x"], v=state["v"])
        if case["drive"]:
            state["lam"], state["plam"] = out["lam"], out["plam"]
        if case["copies"] == 1:  # a sweep reads its statistics only at its end
            abf = [eng.read_abf(*s) for s in state["stages"]]
            for k in ("sum", "sumsq", "count"):
                out["abf_" + k] = np.concatenate([a[k] for a in abf])
            if case["theta"]:
                theta = [eng.read_theta(*s) for s in state["stages"]]
                for k in ("sum_d2", "sum_d", "sum_sd"):
                    out["theta_" + k] = np.concatenate([a[k].ravel() for a in theta])
        return out
    if case["kind"] == "forces":
        e = state["eng"].energy_forces(0, rebuild=True)
        return {k: e[k] for k in ("terms", "U", "dUdl", "dth", "d2th", "F")}
    if case["kind"] == "gradient":
        x, lam, theta = state["x"], state["lam"], state["theta"]
        u = autograd.energy(state["eng"], 0, x, lam, theta)
        gx, gl, gt = torch.autograd.grad(u, (x, lam, theta))
        return dict(U=u.detach(), x=gx, lam=gl, theta=gt)
    f, o = labf.alch_pairs_static(*state["args"], forces=state["forces"], out=state["out"])
    return dict(F=f, out=o)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """Flops: 37 per in-cutoff normal pair and step (force), 45 with the
    energy, 100 per alchemical pair.  Bytes: state, parameters and results
    once per pass."""
    def pairs(n, n_alch, box, r_cut):
        near = 4.0 / 3.0 * math.pi * r_cut ** 3 / box ** 3
        return 0.5 * (n - n_alch) ** 2 * near, n_alch * (n - n_alch) * near

    if case["kind"] in ("lj", "water", "complex"):
        if case["kind"] == "lj":
            n = 4 * case["cells"] ** 3
            sizes = [(n + 1, 1, (n / 0.8) ** (1.0 / 3.0), 2.5)]
        elif case["kind"] == "complex":
            n = 3 * case["waters"] + max(64, round(case["waters"] * 3000 / 31000)) + 40
            sizes = [(n, 40, (n / 98.4) ** (1.0 / 3.0), 1.2)]
        else:
            sizes = []
            for w, s in zip(map(int, case["waters"].split(",")), map(int, case["solutes"].split(","))):
                t = _template("water", w, s)
                sizes.append((t.n, s, t.box, t.r_cut))
        flops = nbytes = 0.0
        for n, na, box, rc in sizes:
            normal, alch = pairs(n, na, box, rc)
            reps = case["walkers"] * case["copies"]
            # integrator about 60 flops per atom, bonded terms about 100 per molecule
            flops += reps * case["steps"] * (37.0 * normal + 100.0 * alch + 100.0 * n)
            nbytes += reps * n * (24 + 24 + 24)
        return dict(bytes=nbytes, flops=flops)
    t = _template("water", case["waters"], case["solutes"])
    normal, alch = pairs(t.n, case["solutes"], t.box, t.r_cut)
    if case["kind"] == "static":
        return dict(bytes=t.n * (12 + 12 + 1 + 4 + 12.0), flops=100.0 * alch + 8.0 * t.n * case["solutes"])
    return dict(bytes=t.n * (12 + 12 + 12.0), flops=45.0 * normal + 100.0 * alch + 100.0 * t.n)


# --------------------------------------------------------------------------
# the method in 64 bits
# --------------------------------------------------------------------------
class _Exact64:
    """U, forces and derivatives of one system, plain torch in FP64."""

    def __init__(self, spec):
        self.dev = torch.device("cuda", 0)
        t = lambda a, dt=torch.float64: torch.as_tensor(np.asarray(a), dtype=dt, device=self.dev)  # noqa: E731
        self.spec, self.L, self.rc = spec, spec.box, spec.r_cut
        rc = spec.r_cut
        self.krf = 1.0 / (2.0 * rc ** 3) if spec.eps_rf <= 0 else (spec.eps_rf - 1.0) / ((2.0 * spec.eps_rf + 1.0) * rc ** 3)
        self.crf = 1.0 / rc + self.krf * rc ** 2
        al = np.asarray(spec.alch) != 0
        self.env, self.alch = t(np.nonzero(~al)[0], torch.long), t(np.nonzero(al)[0], torch.long)
        self.q, self.sig, self.eps = t(spec.charge), t(spec.sigma), t(spec.epsilon)
        self.group, self.extra = t(spec.excl_group, torch.long), t(spec.excl_extra, torch.long)
        self.has_extra = bool((np.asarray(spec.excl_extra) >= 0).any())
        self.mass = t(spec.mass)
        self.bond, self.r0, self.kb = t(spec.bond_ij, torch.long).reshape(-1, 2), t(spec.bond_r0), t(spec.bond_k)
        self.angle, self.t0, self.ka = t(spec.angle_ijk, torch.long).reshape(-1, 3), t(spec.angle_t0), t(spec.angle_k)
        self.pr, self.pr0 = t(spec.posres_idx, torch.long), t(spec.posres_x0).reshape(-1, 3)
        self.fba, self.fbb = t(spec.fb_a, torch.long), t(spec.fb_b, torch.long)

    def mi(self, d):
        return d - self.L * torch.round(d / self.L)

    def kept(self, rows, cols):
        """Pairs (atom of rows, atom of cols) that are not excluded."""
        g = self.group[rows][:, None]
        ok = ~((g >= 0) & (g == self.group[cols][None, :]))
        if self.has_extra:
            for k in range(self.extra.shape[1]):
                ok &= self.extra[rows, k][:, None] != cols[None, :]
                ok &= self.extra[cols, k][None, :] != rows[:, None]
        return ok

    def normal(self, x):
        """Energies and forces of the normal pairs, row blocks of the full matrix."""
        F = torch.zeros_like(x)
        lj = rf = 0.0
        e, s = self.env, self.spec
        block = max(1, 4_000_000 // max(1, len(e)))
        for b in range(0, len(e), block):
            r = e[b:b + block]
            d = self.mi(x[r][:, None, :] - x[e][None, :, :])
            r2 = (d * d).sum(-1)
            ok = self.kept(r, e) & (r2 < self.rc ** 2) & (r[:, None] != e[None, :])
            r2 = torch.where(ok, r2, torch.ones_like(r2))
            qq = s.coul * self.q[r][:, None] * self.q[e][None, :]
            e4 = 4.0 * torch.sqrt(self.eps[r][:, None] * self.eps[e][None, :])
            s6 = ((0.5 * (self.sig[r][:, None] + self.sig[e][None, :])) ** 2 / r2) ** 3
            ri = torch.rsqrt(r2)
            f = (e4 * s6 * (12.0 * s6 - 6.0) + qq * ri) / r2 - 2.0 * self.krf * qq
            f = torch.where(ok, f, torch.zeros_like(f))
            F[r] += (f[..., None] * d).sum(1)
            lj += 0.5 * float(torch.where(ok, e4 * s6 * (s6 - 1.0), torch.zeros_like(f)).sum())
            rf += 0.5 * float(torch.where(ok, qq * (ri + self.krf * r2 - self.crf), torch.zeros_like(f)).sum())
        return lj, rf, F

    def path(self, lam):
        """(lambda_v, lambda_e) of lambda."""
        s = self.spec
        return (torch.where(lam < s.b_v, lam / s.b_v, torch.ones_like(lam)),
                torch.where(lam > s.b_e, (lam - s.b_e) / (1.0 - s.b_e), torch.zeros_like(lam)))

    def alchemical(self, x, lv, le, theta):
        """Soft-core LJ and lambda_e-scaled RF energies (differentiable)."""
        s = self.spec
        a, e = self.alch, self.env
        if len(a) == 0:
            return x.sum() * 0.0, x.sum() * 0.0
        d = self.mi(x[a][:, None, :] - x[e][None, :, :])
        r2 = (d * d).sum(-1)
        ok = self.kept(a, e) & (r2 < self.rc ** 2)
        r2 = torch.where(ok, r2, torch.ones_like(r2))
        rf = (s.coul * theta[:, 2:3] * self.q[e][None, :] * (torch.rsqrt(r2) + self.krf * r2 - self.crf) * ok).sum()
        lj_on = ok & (self.eps[e][None, :] > 0)
        e4 = 4.0 * torch.sqrt(theta[:, 0:1]) * torch.sqrt(self.eps[e])[None, :]
        sg = 0.5 * (theta[:, 1:2] + self.sig[e][None, :])
        soft = s.sc_alpha * (1.0 - lv) ** s.sc_m + (r2 / sg ** 2) ** 3
        sc = (lv ** s.sc_n * e4 * (soft ** -2 - soft ** -1) * lj_on).sum()
        return sc, le * rf

    def bonded(self, x):
        zero = x.sum() * 0.0
        b = a = r = zero
        if len(self.bond):
            d = self.mi(x[self.bond[:, 0]] - x[self.bond[:, 1]])
            b = (0.5 * self.kb * (d.norm(dim=1) - self.r0) ** 2).sum()
        if len(self.angle):
            u = self.mi(x[self.angle[:, 0]] - x[self.angle[:, 1]])
            w = self.mi(x[self.angle[:, 2]] - x[self.angle[:, 1]])
            th = torch.atan2(torch.linalg.cross(u, w).norm(dim=1), (u * w).sum(1))
            a = (0.5 * self.ka * (th - self.t0) ** 2).sum()
        if len(self.pr):
            r = r + 0.5 * self.spec.posres_k * (self.mi(x[self.pr] - self.pr0) ** 2).sum()
        if len(self.fba) and len(self.fbb):
            com = []
            for g in (self.fba, self.fbb):
                w = self.mass[g][:, None]
                com.append(x[g[0]] + (w * self.mi(x[g] - x[g[0]])).sum(0) / w.sum())
            ex = (self.mi(com[0] - com[1]).norm() - self.spec.fb_d0).clamp(min=0.0)
            r = r + 0.5 * self.spec.fb_k * ex ** 2
        return b, a, r

    def all(self, x, lam, derivatives=False):
        """terms (engine order), F, dU/dlambda and, on request, the
        derivatives by (epsilon, sigma, q) of the alchemical atoms."""
        x = x.detach().clone().requires_grad_(True)
        lam = torch.tensor(float(lam), dtype=torch.float64, device=self.dev, requires_grad=True)
        th = torch.stack([self.eps[self.alch], self.sig[self.alch], self.q[self.alch]], 1).requires_grad_(True)
        lj, rf, F = self.normal(x.detach())
        sc, sr = self.alchemical(x, *self.path(lam), th)
        b, a, r = self.bonded(x)
        inputs = [x, lam, th] if len(self.alch) else [x]
        g = torch.autograd.grad(sc + sr + b + a + r, inputs, create_graph=derivatives and len(self.alch) > 0,
                                allow_unused=True)
        out = dict(terms=np.array([lj, rf] + [float(t) for t in (sc, sr, b, a, r)]), F=F - g[0].detach(),
                   dUdl=float(g[1]) if len(self.alch) else 0.0)
        if derivatives:
            out["dth"] = g[2].detach()
            d2 = torch.autograd.grad(g[1], th, allow_unused=True)[0] if g[1].requires_grad else None
            out["d2th"] = torch.zeros_like(th) if d2 is None else d2
        return out


def _philox(c, k0, k1):
    """Philox4x32-10 of counters c (4 uint64 arrays of 32-bit words)."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.asarray(v, np.uint64) for v in c]
    for r in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        ka, kb = np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF), np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF)
        c = [(b >> np.uint64(32)) ^ c[1] ^ ka, b & m, (a >> np.uint64(32)) ^ c[3] ^ kb, a & m]
    return [np.asarray(v) for v in c]


def _normals(seed, walker, step, n, tag):
    z = np.zeros(n, np.uint64)
    r = _philox([np.arange(n, dtype=np.uint64), z + np.uint64(step), z, z + np.uint64(tag)], seed & 0xFFFFFFFF, walker)
    u = [(v >> np.uint64(8)).astype(np.float64) for v in r]
    ra, rb = (np.sqrt(-2.0 * np.log((w + 1.0) / 2 ** 24)) for w in (u[0], u[2]))
    pa, pb = 2.0 * np.pi * u[1] / 2 ** 24, 2.0 * np.pi * u[3] / 2 ** 24
    return np.stack([ra * np.cos(pa), ra * np.sin(pa), rb * np.cos(pb)], 1)


def _exact_md(case, systems):
    """`steps` BAOAB steps of every walker with the ABF fold of each step."""
    out = dict(x=[], v=[], lam=[], plam=[], step=[], abf_sum=[], abf_sumsq=[], abf_count=[])
    th_out = dict(theta_sum_d2=[], theta_sum_d=[], theta_sum_sd=[])
    for spec, run, state in systems:
        E = _Exact64(spec)
        dev, dt, kT = E.dev, run.dt, run.kT
        c, cl = math.exp(-run.gamma * dt), math.exp(-run.gamma_lambda * dt)
        sl = math.sqrt((1.0 - cl * cl) * run.m_lambda * kT)
        sd = torch.sqrt(kT / E.mass)[:, None] * math.sqrt(1.0 - c * c)
        im = 1.0 / E.mass[:, None]
        W = run.n_walkers
        stage = run.walker_stage()
        st = run.stages
        x = [torch.as_tensor(state.x[w], dtype=torch.float64, device=dev) for w in range(W)]
        v = [torch.as_tensor(state.v[w], dtype=torch.float64, device=dev) for w in range(W)]
        lam, plam = state.lam.astype(np.float64).copy(), state.plam.astype(np.float64).copy()
        P = 3 * spec.n_alch + 1
        abf = [np.zeros((3, s.n_bins)) for s in st]
        th = [np.zeros((3, s.n_bins, P)) for s in st]
        ef = [E.all(x[w], lam[w]) for w in range(W)]
        F, G = [e["F"] for e in ef], np.array([-e["dUdl"] for e in ef])

        def bin_of(w):
            s = st[stage[w]]
            return min(max(int(math.floor((lam[w] - s.lo) / ((s.hi - s.lo) / s.n_bins))), 0), s.n_bins - 1)

        def drift(w):
            s = st[stage[w]]
            lam[w] += 0.5 * dt * plam[w] / run.m_lambda
            while lam[w] < s.lo or lam[w] > s.hi:
                lam[w] = 2.0 * (s.lo if lam[w] < s.lo else s.hi) - lam[w]
                plam[w] = -plam[w]

        for k in range(case["steps"]):
            sample, deriv = np.zeros(W), []
            for w in range(W):
                z = torch.as_tensor(_normals(run.seed, w, k, spec.n, 0), device=dev)
                v[w] = v[w] + 0.5 * dt * im * F[w]
                x[w] = x[w] + 0.5 * dt * v[w]
                v[w] = c * v[w] + sd * z
                x[w] = x[w] + 0.5 * dt * v[w]
                plam[w] += 0.5 * dt * G[w]
                drift(w)
                plam[w] = cl * plam[w] + sl * _normals(run.seed, w, k, 1, 1)[0, 0]
                drift(w)
                e = E.all(x[w], lam[w], derivatives=run.theta_stats)
                F[w], sample[w] = e["F"], e["dUdl"]
                v[w] = v[w] + 0.5 * dt * im * F[w]
                if run.theta_stats:
                    deriv.append([np.append(t.cpu().numpy().ravel(), 0.0) for t in (e["dth"], e["d2th"])])
            for w in range(W):
                b = bin_of(w)
                abf[stage[w]][:, b] += (sample[w], sample[w] ** 2, 1.0)
                if run.theta_stats:
                    th[stage[w]][0, b] += deriv[w][1]
                    th[stage[w]][1, b] += deriv[w][0]
                    th[stage[w]][2, b] += sample[w] * deriv[w][0]
            for w in range(W):
                s1, _, n = abf[stage[w]][:, bin_of(w)]
                G[w] = -sample[w] + (min(1.0, n / run.n_full) * s1 / n if n > 0 else 0.0)
                plam[w] += 0.5 * dt * G[w]
        # positions are compared as the engine holds them: wrapped at its own
        # list rebuilds, so only unwrapped-invariant outputs have a value here
        out["v"] += [t.cpu().numpy() for t in v]
        out["lam"].append(lam)
        out["plam"].append(plam)
        for s in range(len(st)):
            for q, key in enumerate(("abf_sum", "abf_sumsq", "abf_count")):
                out[key].append(abf[s][q])
            for q, key in enumerate(th_out):
                th_out[key].append(th[s][q].ravel())
    res = {k: np.concatenate(v) for k, v in out.items() if v}
    res["x"], res["step"] = None, None
    if case["copies"] > 1:
        for k in ("abf_sum", "abf_sumsq", "abf_count"):
            res.pop(k)
    else:
        res["abf_count"] = None
        if case["theta"]:
            res.update({k: np.concatenate(v) for k, v in th_out.items()})
    return res


def exact(case, seed):
    if case["kind"] in ("lj", "water", "complex"):
        if case["kind"] == "complex":
            atoms = [(3.1 * case["waters"], 1)]
        elif case["kind"] == "lj":
            atoms = [(4 * case["cells"] ** 3, 1)]
        else:
            atoms = [(3 * int(w), case["copies"]) for w in case["waters"].split(",")]
        # O(N^2) work in 64 bits, and the host side of every walker step
        evals = case["walkers"] * (case["steps"] + 1)
        if evals * sum(n * n * k for n, k in atoms) > 3e10 or evals * sum(k for _, k in atoms) > 1000:
            return None
        return _exact_md(case, _systems(case, seed))
    spec, _, state = _one_walker(case, seed)
    E = _Exact64(spec)
    x, lam = torch.as_tensor(spec.x, dtype=torch.float64, device=E.dev), float(state.lam[0])
    if case["kind"] == "static":
        l64 = torch.tensor(lam, dtype=torch.float64, device=E.dev, requires_grad=True)
        lv, le = E.path(l64)
        slope = [0.0 if g is None else float(g) for g in
                 (torch.autograd.grad(t, l64, allow_unused=True)[0] for t in (lv, le))]
        th = torch.stack([E.eps[E.alch], E.sig[E.alch], E.q[E.alch]], 1)
        F, every, parts = torch.zeros_like(x), E.alch, np.zeros(4)
        for b in range(0, len(every), 8):  # a few alchemical atoms at a time
            E.alch = every[b:b + 8]
            xb, v, e = (t.detach().clone().requires_grad_(True) for t in (x, lv, le))
            sc, sr = E.alchemical(xb, v, e, th[b:b + 8])
            gx, = torch.autograd.grad(sc + sr, xb, retain_graph=True)
            dv, = torch.autograd.grad(sc, v)
            de, = torch.autograd.grad(sr, e)
            F -= gx
            parts += [float(t) for t in (dv, de, sc, sr)]
        return dict(F=F, out=np.array([slope[0] * parts[0] + slope[1] * parts[1], *parts, 0.0]))
    e = E.all(x, lam, derivatives=True)
    if case["kind"] == "gradient":
        return dict(U=float(e["terms"].sum()), x=-e["F"], lam=e["dUdl"], theta=e["dth"])
    pad = lambda t: np.append(t.cpu().numpy().ravel(), 0.0)  # noqa: E731
    return dict(terms=e["terms"], U=float(e["terms"].sum()), dUdl=e["dUdl"], dth=pad(e["dth"]), d2th=pad(e["d2th"]),
                F=e["F"])
