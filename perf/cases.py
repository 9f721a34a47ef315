"""Measured workloads of the replica engine: what a path-sampling user has it do, through
the public entry points.

Sizes are those of the benchmark and the tests (304-, 560- and 1200-atom chains, the
24 560-site and the 6400-site box, the 256-replica double well, the 512-replica funnel) and,
in `draw`, anything between a 17-atom chain and the largest of them, odd sizes included
(a chain of n atoms is the first n atoms of a generated one).

kinds
  chain   one scps_step_replicas call on chain replicas, then the state on the host: one
          segment of a trajectory between two checkpoints
  scps    the whole self-consistent iteration on a chain (run_chain_scps)
  frames  energies, forces and z of stored frames (post-processing of paths)
  hessian U, its gradient and a Hessian-vector product of a few frames through autograd
  action  sum_t |grad U|^2 over a path and its gradient (checkpointed segments)
  box     a segment of the solvated periodic box
  toy     a segment of the double well
  funnel  the whole self-consistent iteration on the two-dimensional funnel
"""
import dataclasses
import math

import numpy as np
import torch

import paper_1705_02180_gb300 as pkg
import synth
from paper_1705_02180_gb300 import autograd, scps

KT = 0.0083144626 * 300.0
ELEC = {"ddiel": pkg.ELEC_DDIEL, "rf": pkg.ELEC_RF, "plain": pkg.ELEC_PLAIN, "none": pkg.ELEC_NONE}
DT, GAMMA, R0, K_R = 0.002, 1.0, 0.75, 1e-4


# ------------------------------------------------------------------------ cases
def listed():
    return [
        # the double well of the toy section: 256 replicas x 1e4 steps, as the paper-scale run
        {"name": "toy_256", "kind": "toy", "replicas": 256, "steps": 10000},
        # the funnel section as a whole: rMD round, two tube rounds, averages and ranking
        {"name": "funnel_scps", "kind": "funnel", "replicas": 512, "steps": 2000, "save": 20,
         "iterations": 2},
        # the headline workload: 64 Fip35-size chains, one checkpoint segment of 1 ps
        {"name": "chain_64x560", "kind": "chain", "groups": "560:64", "elec": "ddiel",
         "bias": "contacts", "slices": 0, "steps": 500},
        # a lone trajectory in short segments (a user's first run): latency of one replica
        {"name": "chain_1x304", "kind": "chain", "groups": "304:1", "elec": "rf",
         "bias": "contacts", "slices": 0, "steps": 50},
        # uneven batch of three protein sizes in one launch
        {"name": "chain_mixed_512", "kind": "chain", "groups": "304:171,560:171,1200:170",
         "elec": "ddiel", "bias": "contacts", "slices": 0, "steps": 100},
        # the self-consistent rounds: the same chains on the tube variables of 72 maps
        {"name": "chain_tube_64x560", "kind": "chain", "groups": "560:64", "elec": "ddiel",
         "bias": "tube", "slices": 72, "steps": 200},
        # the chain driver end to end with its default 20 replicas, short paths
        {"name": "chain_scps_20x560", "kind": "scps", "atoms": 560, "replicas": 20,
         "steps": 300, "save": 15},
        # post-processing: energies, forces and z of a stored path of 1000 frames
        {"name": "frames_1000x560", "kind": "frames", "atoms": 560, "frames": 1000,
         "elec": "ddiel"},
        # second derivatives at a handful of frames of a large, odd-sized chain
        {"name": "hessian_3x1199", "kind": "hessian", "atoms": 1199, "frames": 3,
         "elec": "plain"},
        # gradient of the action term over a path, checkpointed every 50 frames
        {"name": "action_1000x560", "kind": "action", "atoms": 560, "frames": 1000,
         "segment": 50, "elec": "ddiel"},
        # the solvated box: 16 replicas, one saved frame per 100 steps
        {"name": "box_16x24560", "kind": "box", "residues": 35, "solvent": 24000,
         "replicas": 16, "steps": 100, "save": 100},
        # a small box with two replicas: few tiles, short segments with a checkpoint
        {"name": "box_2x6400", "kind": "box", "residues": 4, "solvent": 6336, "replicas": 2,
         "steps": 50, "save": 0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["toy", "funnel", "chain", "chain", "chain", "chain", "scps", "frames",
                       "hessian", "action", "box"])
    elec = rng.choice(["ddiel", "ddiel", "rf", "plain", "none"])
    if kind == "toy":
        return {"kind": kind, "replicas": _log(rng, 1, 512), "steps": _log(rng, 50, 9000)}
    if kind == "funnel":
        save = _log(rng, 5, 40)
        return {"kind": kind, "replicas": _log(rng, 64, 500), "steps": save * rng.randint(400 // save, 1500 // save),
                "save": save, "iterations": rng.choice([1, 2])}
    if kind == "chain":
        groups, total = [], 0
        for _ in range(rng.choice([1, 1, 2, 3])):
            n = _log(rng, 17, 1200)
            r = max(1, min(_log(rng, 1, 256), 120000 // n))
            groups.append("%d:%d" % (n, r))
            total += n * r
        bias = rng.choice(["contacts", "contacts", "tube", "none"])
        return {"kind": kind, "groups": ",".join(groups), "elec": elec, "bias": bias,
                "slices": _log(rng, 3, 128) if bias == "tube" else 0,
                "steps": max(5, min(_log(rng, 10, 500), 20000000 // total))}
    if kind == "scps":
        save = _log(rng, 5, 40)
        return {"kind": kind, "atoms": _log(rng, 150, 560), "replicas": _log(rng, 2, 20),
                "steps": save * rng.randint(4, 20), "save": save}
    if kind == "frames":
        n = _log(rng, 17, 1200)
        return {"kind": kind, "atoms": n, "frames": min(_log(rng, 1, 1500), 500000 // n), "elec": elec}
    if kind == "hessian":
        return {"kind": kind, "atoms": _log(rng, 17, 1200), "frames": _log(rng, 1, 40), "elec": elec}
    if kind == "action":
        n = _log(rng, 64, 800)
        return {"kind": kind, "atoms": n, "frames": min(_log(rng, 20, 900), 400000 // n),
                "segment": rng.choice([20, 50, 50, 100]), "elec": elec}
    res = rng.choice([4, 19, 35])
    sites = _log(rng, {4: 5000, 19: 8000, 35: 14000}[res], 22000)
    return {"kind": "box", "residues": res, "solvent": sites,
            "replicas": rng.randint(1, max(1, 120000 // sites)), "steps": _log(rng, 10, 60), "save": 0}


# ------------------------------------------------------------------------ inputs
_made = {}


def _once(key, make):
    if key not in _made:
        _made[key] = make()
    return _made[key]


def _generated(n_res):
    def make():
        try:
            return synth.make_chain(n_res, seed=1)
        except OSError:  # a read-only tree: no generator cache
            return synth.make_chain(n_res, seed=1, cache=False)
    return _once(("chain", n_res), make)


def _chain(n):
    """The first n atoms of the smallest generated chain that has them."""
    def make():
        c = _generated(next(r for r in (4, 19, 35, 75) if 16 * r >= n))
        if n == c.n_atoms:
            return c
        kb, ka = (c.bonds < n).all(1), (c.angles < n).all(1)
        return dataclasses.replace(
            c, n_atoms=n, mass=c.mass[:n], charge=c.charge[:n], sigma=c.sigma[:n], eps=c.eps[:n],
            bonds=c.bonds[kb], b0=c.b0[kb], kb=c.kb[kb], angles=c.angles[ka], th0=c.th0[ka],
            kth=c.kth[ka], exclusions=c.exclusions[(c.exclusions < n).all(1)],
            x_native=c.x_native[:n], x_unfolded=c.x_unfolded[:n],
            contacts=c.contacts[(c.contacts < n).all(1)])
    return _once(("cut", n), make)


def _f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def _groups(case):
    return [tuple(int(v) for v in g.split(":")) for g in case["groups"].split(",")]


def _bias(case, chains):
    """The bias a chain case runs with: chains without a native contact have none."""
    return case["bias"] if all(len(c.contacts) for c in chains) else "none"


def _maps(c, K):
    """Reference maps (K, contacts) along contact distances going from X_U to X_N."""
    d = [np.linalg.norm(x[c.contacts[:, 1]] - x[c.contacts[:, 0]], axis=1) for x in (c.x_unfolded, c.x_native)]
    r = d[0][None] + (d[1] - d[0])[None] * np.linspace(0.0, 1.0, K)[:, None]
    u = (r / R0) ** 2
    return (1 + u + u * u) / (1 + u + u * u + u ** 3 + u ** 4)


TUBE = {"lam": 13.5, "k_s": 2.5, "k_w": 2.5e-4}


def _chain_inputs(case, seed):
    gs = _groups(case)
    chains = [_chain(n) for n, _ in gs]
    x = [np.broadcast_to(_f32(c.x_unfolded), (r, c.n_atoms, 3)) for c, (_, r) in zip(chains, gs)]
    v = [_f32(c.velocities(r, KT, seed + 1 + k)) for k, (c, (_, r)) in enumerate(zip(chains, gs))]
    return gs, chains, x, v


def _pack(parts):
    return np.concatenate([np.reshape(p, (-1, 3)) for p in parts])


def _frames(c, T, seed):
    """T frames around X_U and X_N in turn, 0.01 nm noise, on the GPU."""
    g = torch.Generator("cuda").manual_seed(seed)
    base = torch.from_numpy(np.stack([c.x_unfolded, c.x_native]).astype(np.float32)).cuda()
    x = base[torch.arange(T, device="cuda") % 2]
    return (x + 0.01 * torch.randn(x.shape, generator=g, device="cuda")).contiguous()


def _evaluator(c, elec):
    return pkg.System(topologies=[pkg.chain_topology(c)], replica_topology=[0], x0=c.x_unfolded,
                      elec=ELEC[elec], dt=DT, gamma=GAMMA, kT=KT, seed=1)


def _box(case):
    """A chain in solvent sites (100 sites/nm^3); every size drawn leaves the chain clear of its
    own images."""
    def make():
        _generated(case["residues"])
        try:
            return synth.make_box(case["residues"], case["solvent"], seed=1)
        except OSError:
            return synth.make_box(case["residues"], case["solvent"], seed=1, cache=False)
    return _once(("box", case["residues"], case["solvent"]), make)


def _box_inputs(case, seed):
    b = _box(case)
    return b, _f32(b.x), _f32(b.velocities(case["replicas"], KT, seed))


# ------------------------------------------------------------------------ prepare / run
def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "toy":
        t = synth.make_toy(case["replicas"])
        s = pkg.System(model=pkg.MODEL_TOY2D, x0=t.start_positions(), integrator=pkg.INT_EM, dt=t.dt,
                       gamma=t.gamma, kT=t.kT, seed=seed)
        s.set_toy_bias(t.k_R, x_ref=1.0)
        st["system"] = s
    elif kind == "funnel":
        st["protocol"] = _funnel(case, seed)
    elif kind == "chain":
        gs, chains, x, v = _chain_inputs(case, seed)
        reps = np.concatenate([np.full(r, k) for k, (_, r) in enumerate(gs)])
        s = pkg.System(topologies=[pkg.chain_topology(c) for c in chains], replica_topology=reps,
                       x0=_pack(x), v0=_pack(v), elec=ELEC[case["elec"]], dt=DT, gamma=GAMMA, kT=KT,
                       seed=seed)
        bias = _bias(case, chains)
        if bias == "contacts":
            s.set_contact_bias([c.contacts for c in chains], [c.x_native for c in chains], k_R=K_R, r0=R0)
        elif bias == "tube":
            K = case["slices"]
            t = (np.arange(K) + 1) * 7.0
            s.set_contact_tube_bias([c.contacts for c in chains], [c.x_native for c in chains],
                                    [_maps(c, K) for c in chains], t, TUBE["lam"], TUBE["k_s"],
                                    TUBE["k_w"], t[-1], r0=R0)
        st["system"] = s
    elif kind == "scps":
        st["chain"] = _chain(case["atoms"])
        st["protocol"] = _chain_protocol(case, seed)
    elif kind in ("frames", "hessian", "action"):
        c = _chain(case["atoms"])
        s = _evaluator(c, case["elec"])
        st.update(system=s, X=_frames(c, case["frames"], seed), z=False)
        T = case["frames"]
        if kind == "frames":
            st["z"] = len(c.contacts) > 0
            if st["z"]:
                s.set_contact_bias([c.contacts], [c.x_native], k_R=K_R, r0=R0)
            st["U"] = torch.empty(T, dtype=torch.float64, device="cuda")
            st["Z"] = torch.empty_like(st["U"])
            st["F"] = torch.empty_like(st["X"])
        if kind == "hessian":
            st["V"] = _direction(st["X"], seed)
    else:
        b, x, v = _box_inputs(case, seed)
        R, save = case["replicas"], case["save"]
        s = pkg.System(topologies=[b.topology()], replica_topology=[0] * R,
                       x0=np.broadcast_to(x, (R,) + x.shape).reshape(-1, 3), v0=v.reshape(-1, 3), cutoff=1.0,
                       elec=pkg.ELEC_RF, eps_rf=78.5, box=b.box, dt=DT, gamma=GAMMA, kT=KT, seed=seed,
                       save_interval=save, max_frames=1 if save else 0)
        if len(b.chain.contacts):
            s.set_contact_bias([b.chain.contacts], [b.chain.x_native], k_R=K_R, r0=R0)
        st["system"] = s
    return st


def _direction(X, seed):
    g = torch.Generator("cuda").manual_seed(seed + 77)
    return torch.randn(X.shape, generator=g, device="cuda")


def _funnel(case, seed):
    return scps.FunnelProtocol(n_replicas=case["replicas"], n_steps=case["steps"],
                               save_every=case["save"], iterations=case["iterations"], seed=seed)


def _chain_protocol(case, seed):
    # z_native 2: paths this short end near their start, all of them go into the averages
    return scps.ChainProtocol(n_replicas=case["replicas"], kT=KT, n_steps=case["steps"],
                              save_every=case["save"], z_native=2.0, iterations=1, seed=seed)


def run(st):
    kind, case = st["kind"], st["case"]
    s = st.get("system")
    if kind in ("toy", "chain") or (kind == "box" and not case["save"]):
        s.step(case["steps"])
        return s.get_state()
    if kind == "box":
        s.step(case["steps"])
        paths = s.collect_paths()
        return {k: np.stack([p[k] for p in paths]) for k in paths[0]}
    if kind == "funnel":
        return _scps_outputs(scps.run_funnel_scps(st["protocol"]))
    if kind == "scps":
        return _scps_outputs(scps.run_chain_scps(st["chain"], st["protocol"]))
    if kind == "frames":
        s.energy_forces(0, st["X"], st["U"], st["F"], st["Z"] if st["z"] else None)
        return {"U": st["U"], "F": st["F"], "z": st["Z"]} if st["z"] else {"U": st["U"], "F": st["F"]}
    X = st["X"].detach().requires_grad_(True)
    if kind == "hessian":
        U = autograd.potential_energy(s, X)
        (G,) = torch.autograd.grad(U.sum(), X, create_graph=True)
        (HV,) = torch.autograd.grad(G, X, st["V"])
        return {"U": U.detach(), "G": G.detach(), "HV": HV}
    A = autograd.force_norm_action(s, X, segment=case["segment"])
    A.backward()
    return {"A": A.detach(), "grad": X.grad}


def _scps_outputs(res):
    out = {"times": res["times"]}
    for k, r in enumerate(res["rounds"]):
        out["round%d" % k] = {q: np.asarray(r[q]) for q in ("T", "ref", "maps") if q in r}
        out["round%d" % k]["reactive"] = np.isin(np.arange(len(r["T"])), r["reactive"])
    for q in ("best", "best_path"):
        if q in res:
            out[q] = res[q]
    return out


# ------------------------------------------------------------------------ work
def _pairs(n):
    """In-cutoff pairs of an n-atom chain (43.6k at 560 atoms, thermally unfolded)."""
    return n * min(0.5 * (n - 1), 17.0 * n ** 0.24)


def _chain_flops(c):
    return 49 * _pairs(c.n_atoms) + 20 * len(c.bonds) + 60 * len(c.angles) + 40 * c.n_atoms


def work(case):
    kind = case["kind"]
    if kind == "toy":
        return {"bytes": 80.0 * case["replicas"], "flops": 60.0 * case["replicas"] * case["steps"]}
    if kind == "funnel":
        n, K = case["replicas"] * case["steps"], case["steps"] // case["save"]
        rounds = 1 + case["iterations"]
        return {"bytes": rounds * case["replicas"] * (80.0 + 40.0 * K),
                "flops": n * (90.0 * rounds + 20.0 * K * case["iterations"])}
    if kind == "chain":
        gs = _groups(case)
        chains = [_chain(n) for n, _ in gs]
        bias = _bias(case, chains)
        fl = by = 0.0
        for c, (n, r) in zip(chains, gs):
            per = {"none": 0, "contacts": 30, "tube": 20 + 5 * case["slices"]}[bias] * len(c.contacts)
            fl += r * case["steps"] * (_chain_flops(c) + per)
            by += r * n * 96.0 + (4.0 * case["slices"] * len(c.contacts) if bias == "tube" else 0)
        return {"bytes": by, "flops": fl}
    if kind == "scps":
        c, K = _chain(case["atoms"]), case["steps"] // case["save"]
        n = case["replicas"] * case["steps"]
        return {"bytes": 2 * case["replicas"] * c.n_atoms * (48.0 + 12.0 * K) + 8.0 * K * len(c.contacts),
                "flops": n * (2 * _chain_flops(c) + (50 + 5 * K) * len(c.contacts))}
    if kind in ("frames", "hessian", "action"):
        c, T = _chain(case["atoms"]), case["frames"]
        hv = 70 * _pairs(c.n_atoms)
        return {"frames": {"bytes": T * (24.0 * c.n_atoms + 16), "flops": T * (_chain_flops(c) + 30 * len(c.contacts))},
                "hessian": {"bytes": T * (48.0 * c.n_atoms + 8), "flops": T * (_chain_flops(c) + hv)},
                "action": {"bytes": T * 24.0 * c.n_atoms, "flops": T * (_chain_flops(c) + hv)}}[kind]
    n = 16 * case["residues"] + case["solvent"]
    return {"bytes": 100.0 * n * case["replicas"],
            "flops": case["replicas"] * case["steps"] * n * (209 * 49.0 + 40)}


# ------------------------------------------------------------------------ exact values
# Plain torch / numpy in 64 bits: every non-excluded pair of a chain (all pairs within the
# cutoff sphere of the box), sums and square roots as they come.
COULOMB = 138.935458


class _Field:
    """-grad U, U, z and the tube variables of one chain for a batch of configurations."""

    def __init__(self, c, elec, box=0.0, dev="cuda", solvent=None):
        t = lambda a, **k: torch.as_tensor(np.ascontiguousarray(a), device=dev, **k)  # noqa: E731
        src = solvent or c
        self.n, self.elec, self.box = len(src.mass), elec, box
        self.mass = t(src.mass)
        self.sigma, self.eps, self.q = t(src.sigma), t(src.eps), t(src.charge)
        ij = torch.triu_indices(self.n, self.n, 1, device=dev)
        ok = torch.ones(self.n, self.n, dtype=torch.bool, device=dev)
        if len(c.exclusions):
            e = t(c.exclusions.astype(np.int64))
            ok[e[:, 0], e[:, 1]] = False
            ok[e[:, 1], e[:, 0]] = False
        self.ij = ij[:, ok[ij[0], ij[1]]]
        self.bonds, self.b0, self.kb = t(c.bonds.astype(np.int64)), t(c.b0), t(c.kb)
        self.ang, self.th0, self.kth = t(c.angles.astype(np.int64)), t(c.th0), t(c.kth)
        self.con = t(c.contacts.astype(np.int64).reshape(-1, 2))
        xn = t(c.x_native)
        if len(c.contacts):
            self.C0 = self._C(((xn[self.con[:, 1]] - xn[self.con[:, 0]]) ** 2).sum(-1) / R0 ** 2)

    @staticmethod
    def _C(u):
        return (1 + u + u * u) / (1 + u + u * u + u ** 3 + u ** 4)

    def _mi(self, d):
        return d - self.box * torch.round(d / self.box) if self.box else d

    def _phi(self, r2, i, j):
        """Shifted-force pair energy with its -dphi/dr / r (cutoff 1 nm)."""
        sig, eps, qq = 0.5 * (self.sigma[i] + self.sigma[j]), (self.eps[i] * self.eps[j]).sqrt(), self.q[i] * self.q[j]
        r = r2.sqrt()

        def raw(r):
            s6 = (sig / r) ** 6
            e, f = 4 * eps * (s6 * s6 - s6), 24 * eps * (2 * s6 * s6 - s6) / r
            if self.elec == "ddiel":
                k = COULOMB / 40.0 * qq
                return e + k / r ** 2, f + 2 * k / r ** 3
            if self.elec == "rf":
                krf = (78.5 - 1) / (2 * 78.5 + 1)
                return e + COULOMB * qq * (1 / r + krf * r ** 2 - 1 - krf), f + COULOMB * qq * (1 / r ** 2 - 2 * krf * r)
            if self.elec == "plain":
                return e + COULOMB * qq / r, f + COULOMB * qq / r ** 2
            return e, f
        e, f = raw(r)
        ec, fc = raw(torch.ones_like(r))
        return e - ec + (r - 1) * fc, (f - fc) / r

    def bonded(self, x):
        a, b = x[:, self.bonds[:, 0]], x[:, self.bonds[:, 1]]
        e = (0.5 * self.kb * (self._mi(b - a).norm(dim=-1) - self.b0) ** 2).sum(-1)
        p, q, s = (x[:, self.ang[:, k]] for k in range(3))
        u, w = self._mi(p - q), self._mi(s - q)
        th = torch.atan2(torch.linalg.cross(u, w).norm(dim=-1), (u * w).sum(-1))
        return e + (0.5 * self.kth * (th - self.th0) ** 2).sum(-1)

    def energy(self, x):
        """U with autograd through everything (a few frames at a time)."""
        i, j = self.ij
        r2 = (self._mi(x[:, j] - x[:, i]) ** 2).sum(-1)
        near = r2 < 1.0
        e = torch.zeros(x.shape[0], dtype=x.dtype, device=x.device)
        f, p = near.nonzero(as_tuple=True)
        phi, _ = self._phi(r2[f, p], i[p], j[p])
        return e.index_add(0, f, phi) + self.bonded(x)

    def pair_forces(self, x, chunk=24_000_000):
        F = torch.zeros(x.shape, dtype=x.dtype, device=x.device)
        E = torch.zeros(x.shape[0], dtype=x.dtype, device=x.device)
        P = self.ij.shape[1]
        step = max(1, chunk // P)
        for a in range(0, x.shape[0], step):
            xs = x[a:a + step]
            for b in range(0, P, chunk):
                i, j = self.ij[:, b:b + chunk]
                r2 = torch.zeros(xs.shape[0], len(i), dtype=x.dtype, device=x.device)
                for k in range(3):
                    r2 += self._mi(xs[:, j, k] - xs[:, i, k]) ** 2
                f, p = (r2 < 1.0).nonzero(as_tuple=True)
                ii, jj = i[p], j[p]
                e, s = self._phi(r2[f, p], ii, jj)
                d = self._mi(xs[f, jj] - xs[f, ii]) * s[:, None]
                n = self.n
                F[a:a + step].view(-1, 3).index_add_(0, f * n + jj, d).index_add_(0, f * n + ii, -d)
                E[a:a + step].index_add_(0, f, e)
        return F, E

    def forces(self, x):
        F, E = self.pair_forces(x)
        with torch.enable_grad():
            y = x.detach().requires_grad_(True)
            eb = self.bonded(y)
            (g,) = torch.autograd.grad(eb.sum(), y)
        return F - g, E + eb.detach()

    def contacts(self, x):
        d = self._mi(x[:, self.con[:, 1]] - x[:, self.con[:, 0]])
        u = (d * d).sum(-1) / R0 ** 2
        num, den = 1 + u + u * u, 1 + u + u * u + u ** 3 + u ** 4
        dC = ((1 + 2 * u) * den - num * (1 + 2 * u + 3 * u * u + 4 * u ** 3)) / den ** 2
        return d, num / den, dC

    def z(self, x):
        _, C, _ = self.contacts(x)
        return ((C - self.C0) ** 2).sum(-1)

    def contact_gradient(self, x, w):
        """sum_p w_p grad C_p."""
        d, _, dC = self.contacts(x)
        g = d * (w * dC * 2 / R0 ** 2)[..., None]
        G = torch.zeros_like(x)
        return G.index_add_(1, self.con[:, 1], g).index_add_(1, self.con[:, 0], -g)


def _philox(atoms, rep, step, seed):
    """Philox4x32-10 words for counters (atom, replica, step, 0): int64 tensor (R, n, 4)."""
    dev = rep.device
    m = 0xFFFFFFFF
    c = [atoms[None, :].expand(len(rep), -1), rep[:, None].expand(-1, len(atoms)),
         torch.full((len(rep), len(atoms)), step, dtype=torch.int64, device=dev),
         torch.zeros(len(rep), len(atoms), dtype=torch.int64, device=dev)]
    k0, k1 = seed & m, (seed >> 32) & m

    def mul(a, x):  # high and low words of a 32 x 32 bit product
        xl, xh = x & 0xFFFF, x >> 16
        lo = a * xl
        mid = a * xh + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return torch.stack(c, -1)


def _normals(w):
    u = w.double()
    rad = torch.sqrt(-2 * torch.log((u[..., 0::2] + 1) * 2.0 ** -32))
    th = 2 * math.pi * u[..., 1::2] * 2.0 ** -32
    return torch.stack([rad * torch.cos(th), rad * torch.sin(th)], -1).flatten(-2)


def _trajectory(field, x, v, rep, seed, steps, bias, maps=None, times=None, t_path=1.0, save=0):
    """BAOAB with the ratchet (contacts) or the tube forces; returns x, v, zm, T, frames."""
    dev = x.device
    n, R = field.n, x.shape[0]
    im = (1 / field.mass)[None, :, None]
    c1 = math.exp(-GAMMA * DT)
    sd = torch.sqrt((1 - c1 * c1) * KT * im)
    inf = torch.full((R,), math.inf, dtype=torch.float64, device=dev)
    zm, sm, wm, T = inf.clone(), inf.clone(), inf.clone(), torch.zeros_like(inf)
    atoms = torch.arange(n, device=dev)

    def force():
        nonlocal zm, sm, wm
        F, _ = field.forces(x)
        if bias == "none":
            return F, torch.zeros_like(T)
        _, C, _ = field.contacts(x)
        if bias == "contacts":
            z = ((C - field.C0) ** 2).sum(-1)
            fac = torch.where(z < zm, torch.zeros_like(z), -K_R * (z - zm))
            zm = torch.minimum(zm, z)
            w = fac[:, None] * 2 * (C - field.C0)
        else:
            n0 = (field.C0 ** 2).sum()
            D = ((C[:, None, :] - maps[None]) ** 2).sum(-1) / n0
            lam = TUBE["lam"]
            p = torch.softmax(-lam * D, 1)
            wv = -torch.logsumexp(-lam * D, 1) / lam
            tb = (p * times).sum(1)
            sv = 1 - tb / t_path
            cs = torch.where(sv < sm, torch.zeros_like(sv), -TUBE["k_s"] * (sv - sm))
            cw = torch.where(wv < wm, torch.zeros_like(wv), -TUBE["k_w"] * (wv - wm))
            sm, wm = torch.minimum(sm, sv), torch.minimum(wm, wv)
            zm = sm
            gam = cs[:, None] * lam / t_path * p * (times - tb[:, None]) + cw[:, None] * p
            w = 2 / n0 * (C * gam.sum(1, keepdim=True) - gam @ maps)
        B = field.contact_gradient(x, w)
        return F + B, DT / GAMMA * (B * B * im).sum((1, 2))

    F, _ = force()
    frames = []
    for s in range(steps):
        v = v + 0.5 * DT * im * F
        x = x + 0.5 * DT * v
        v = c1 * v + sd * _normals(_philox(atoms, rep, s, seed))[..., :3]
        x = x + 0.5 * DT * v
        F, dT = force()
        T = T + dT
        v = v + 0.5 * DT * im * F
        if save and (s + 1) % save == 0:
            frames.append(x)
    return x, v, zm, T, frames


def _np(t):
    return t.cpu().numpy()


def _exact_chain(case, seed):
    gs, chains, x, v = _chain_inputs(case, seed)
    if sum(r * n * n * 0.5 for n, r in gs) * case["steps"] > 2.2e10:
        return None
    bias, first, parts = _bias(case, chains), 0, []
    for k, (c, (n, r)) in enumerate(zip(chains, gs)):
        f = _Field(c, case["elec"])
        maps = times = None
        t_path = 1.0
        if bias == "tube":
            maps = torch.from_numpy(_maps(c, case["slices"])).cuda()
            times = (torch.arange(case["slices"], device="cuda").double() + 1) * 7.0
            t_path = 7.0 * case["slices"]
        parts.append(_trajectory(f, torch.from_numpy(np.array(x[k])).cuda(), torch.from_numpy(v[k]).cuda(),
                                 torch.arange(first, first + r, device="cuda"), seed, case["steps"], bias,
                                 maps, times, t_path))
        first += r
    cat = lambda q: np.concatenate([_np(p[q]) for p in parts])  # noqa: E731
    # (under the tube bias the state's z_m is not the ratchet's minimum, and T sums squares of
    # s - s_m and w - w_m, differences that short segments leave near the FP32 resolution of s
    # and w, to which the engine holds them)
    return {"x": _pack([_np(p[0]) for p in parts]), "v": _pack([_np(p[1]) for p in parts]),
            "zm": None if bias == "tube" else cat(2), "step": None,
            "T": None if bias == "tube" else cat(3)}


def _exact_scps(case, seed):
    c, R, steps, save = _chain(case["atoms"]), case["replicas"], case["steps"], case["save"]
    if not len(c.contacts) or 1.0 * R * c.n_atoms ** 2 * steps > 2.2e10:
        return None
    f = _Field(c, "ddiel")
    K = steps // save
    times = (torch.arange(K, device="cuda").double() + 1) * save * DT
    x0 = torch.from_numpy(_f32(np.broadcast_to(c.x_unfolded, (R, c.n_atoms, 3)))).cuda()
    rep = torch.arange(R, device="cuda")
    v0 = torch.from_numpy(_f32(c.velocities(R, KT, seed))).cuda()
    _, _, _, T0, frames = _trajectory(f, x0, v0, rep, seed, steps, "contacts", save=save)
    maps = torch.stack([f.contacts(y)[1].mean(0) for y in frames])
    return {"times": _np(times), "round0": {"T": _np(T0), "reactive": None},
            "round1": {"T": None, "maps": _np(maps), "reactive": None}, "best": None}


def _exact_frames(case, seed):
    c, kind = _chain(case["atoms"]), case["kind"]
    f, X = _Field(c, case["elec"]), _frames(c, case["frames"], seed).double()
    if kind == "frames":
        F, U = f.forces(X)
        out = {"U": U, "F": F}
        if len(c.contacts):
            out["z"] = f.z(X)
        return out
    U, G, HV = [], [], []
    step = max(1, 3_000_000 // f.ij.shape[1])
    for a in range(0, len(X), step):
        with torch.enable_grad():
            x = X[a:a + step].requires_grad_(True)
            u = f.energy(x)
            (g,) = torch.autograd.grad(u.sum(), x, create_graph=True)
            w = _direction(X, seed)[a:a + step].double() if kind == "hessian" else 2 * g.detach()
            (h,) = torch.autograd.grad(g, x, w)
        U.append(u.detach())
        G.append(g.detach())
        HV.append(h)
    U, G, HV = torch.cat(U), torch.cat(G), torch.cat(HV)
    return {"U": U, "G": G, "HV": HV} if kind == "hessian" else {"A": (G * G).sum(), "grad": HV}


def _exact_box(case, seed):
    b, x, v = _box_inputs(case, seed)
    if case["save"] or 0.5 * b.n_atoms ** 2 * case["replicas"] * case["steps"] > 1.2e10:
        return None
    f = _Field(b.chain, "rf", box=b.box, solvent=b)
    R = case["replicas"]
    # one replica after the other (positions come back in whichever image the last list
    # build left them, so they are not compared)
    parts = [_trajectory(f, torch.from_numpy(x[None]).cuda(), torch.from_numpy(v[r:r + 1]).cuda(),
                         torch.arange(r, r + 1, device="cuda"), seed, case["steps"],
                         "contacts" if len(b.chain.contacts) else "none") for r in range(R)]
    cat = lambda q: np.concatenate([_np(p[q]) for p in parts])  # noqa: E731
    return {"x": None, "v": cat(1).reshape(-1, 3), "zm": cat(2), "step": None, "T": cat(3)}


def _noise2(R, steps, seed):
    """Gaussian pairs (steps, R, 2) of the two-dimensional models (one particle, atom word 0)."""
    out = np.empty((steps, R, 2))
    rep, zero = torch.arange(R), torch.zeros(1, dtype=torch.int64)
    for s in range(steps):
        out[s] = _normals(_philox(zero, rep, s, seed))[:, 0, :2].numpy()
    return out


def _exact_toy(case, seed):
    t, R = synth.make_toy(case["replicas"]), case["replicas"]
    if R * case["steps"] > 1e7:
        return None
    p = t.start_positions()
    zm, T = np.full(R, np.inf), np.zeros(R)
    a, sd = t.dt / t.gamma, math.sqrt(2 * t.kT * t.dt / t.gamma)
    xi = _noise2(R, case["steps"], seed)
    for s in range(case["steps"]):
        x, y = p[:, 0], p[:, 1]
        z = (x - 1) ** 2
        b = np.where(z < zm, 0.0, -t.k_R * (z - np.minimum(z, zm)) * 2 * (x - 1))
        zm = np.minimum(zm, z)
        T += a * b * b
        p = p + a * np.stack([-4 * x * (x * x - 1) + b, -2 * y], 1) + sd * xi[s]
    return {"x": p, "v": np.zeros_like(p), "zm": zm, "step": None, "T": T}


def _funnel_round(p, seed, ref, times):
    R = p.n_replicas
    q = np.tile(np.asarray(p.start, float), (R, 1))
    m = [np.full(R, np.inf), np.full(R, np.inf)]
    T, a, sd = np.zeros(R), p.dt / p.gamma, math.sqrt(2 * p.kT * p.dt / p.gamma)
    xi = _noise2(R, p.n_steps, seed)
    t_path, frames = p.n_steps * p.dt, []

    def ratchet(v, k, which):
        f = np.where(v < m[which], 0.0, -k * (v - np.minimum(v, m[which])))
        m[which] = np.minimum(m[which], v)
        return f[:, None]
    gate = np.array([1.5, 0.0])
    for s in range(p.n_steps):
        r2, d2 = (q * q).sum(1), ((q - gate) ** 2).sum(1)
        gr = -2 * 0.03 ** 2 * r2 - 60 / (r2 + 1) ** 3 + 160 / (r2 + 4) ** 3
        gd = -3 / (d2 + 0.25) ** 3
        f = 2 * (gr[:, None] * q + gd[:, None] * (q - gate))
        if ref is None:
            z = np.sqrt(r2)
            b = ratchet(z, p.k_R, 0) * q / z[:, None]
        else:
            d = q[:, None] - ref[None]
            D = (d * d).sum(-1)
            e = np.exp(-p.lam * (D - D.min(1, keepdims=True)))
            S = e.sum(1)
            pi = e / S[:, None]
            tm = (pi * times).sum(1)
            gw = (pi[..., None] * 2 * d).sum(1)
            gs = p.lam / t_path * ((pi * times)[..., None] * 2 * d).sum(1) - p.lam / t_path * tm[:, None] * gw
            b = ratchet(1 - tm / t_path, p.k_s, 0) * gs + ratchet(D.min(1) - np.log(S) / p.lam, p.k_w, 1) * gw
        T += a * (b * b).sum(1)
        q = q + a * (f + b) + sd * xi[s]
        if (s + 1) % p.save_every == 0:
            frames.append(q)
    return q, T, np.stack(frames, 1)


def _exact_funnel(case, seed):
    p = _funnel(case, seed)
    K = p.n_steps // p.save_every
    if p.n_replicas * p.n_steps * K * p.iterations > 3e8:
        return None
    times = (np.arange(K) + 1) * p.save_every * p.dt
    out, ref = {"times": times}, None
    for it in range(1 + p.iterations):
        q, T, fr = _funnel_round(p, seed + it, ref, times)
        react = np.flatnonzero(np.hypot(q[:, 0], q[:, 1]) < p.r_native)
        out["round%d" % it] = {"reactive": None, "T": T}
        if ref is not None:
            out["round%d" % it]["ref"] = ref
        if not len(react):
            break
        best = fr[react[np.argmin(T[react])]]
        ref = fr[react].mean(0)
    if len(react):
        out["best"], out["best_path"] = None, best
    return out


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "toy":
            return _exact_toy(case, seed)
        if kind == "funnel":
            return _exact_funnel(case, seed)
        if kind == "chain":
            return _exact_chain(case, seed)
        if kind == "scps":
            return _exact_scps(case, seed)
        if kind == "box":
            return _exact_box(case, seed)
        return _exact_frames(case, seed)
