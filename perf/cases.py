"""Performance cases: passes of the Gen. ParRep hot path through the public binding.

Each case is one pass that a user's program makes again and again: an exit test of the convergence step
(`grp_fv_check`, `grp_batch_fv_check`: a BAOAB segment with sampling, the state check, Fleming-Viot
branching, Gelman-Rubin ratios and the status readback), a plain segment (`grp_step_k`), a segment with its
adjoint (`grp_adjoint_segment`) or energies with their gradients (`grp_energy_grad`).  `exact` repeats a pass
in 64-bit torch from the same inputs: its own noise, integrator, energies (forces by automatic
differentiation), sampling, branching and ratios.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1807_02431_gb300 import binding as B
from paper_1807_02431_gb300 import workloads as W

FP64, MIXED = "fp64", "mixed"


# ------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the validation system: one particle in a double well, 32 replicas, an exit test every 100 steps.
        # The smallest call there is: launches, the readback and the serial chain of FP64 steps count.
        dict(name="well_check_r32", kind="well", R=32, k=100),
        # many states, many runs: 64 runs of a 7-bead alkane, 32 replicas each, one batched exit test
        dict(name="alkane_batch_64x32", kind="alkanes", n=7, runs=64, R=32, k=100, precision=MIXED),
        # the headline workload: alanine-dipeptide-like chain, 256 replicas, exit tests every 500 steps
        dict(name="chain22_check_r256", kind="chain", n=22, R=256, k=500, precision=MIXED, check=True),
        # the same system advanced on the FP64 path (the path that a mixed result is checked against)
        dict(name="chain22_step_r256_fp64", kind="chain", n=22, R=256, k=500, precision=FP64, check=False),
        # hydrogens with constrained bonds, as molecular dynamics setups run them (exit tests every 200 steps: the
        # hydrogens' motion loses its first digit against 64 bits after about 300)
        dict(name="chain22h_check_r256", kind="chain_h", n=22, R=256, k=200, precision=MIXED, check=True),
        # the chain in implicit solvent (OBC II)
        dict(name="chain22_solvent_r256", kind="solvated", n=22, R=256, k=500, precision=MIXED, check=True),
        # a periodic box with ions: particle mesh Ewald and Verlet lists, 220 atoms
        dict(name="ions220_step_r256", kind="ions", n=100, pairs=60, edge=4.0, R=256, k=500, precision=MIXED,
             check=False),
        # batched runs of chains of very uneven sizes (22 to 400 beads)
        dict(name="chains_batch_64x128", kind="chains", runs=64, R=128, lo=22, hi=400, k=500, precision=MIXED),
        # ligand in the pocket of a 2,000-bead receptor, 1,024 replicas: the largest system
        dict(name="ligand_check_r1024", kind="ligand", n=2000, R=1024, k=500, precision=MIXED, check=True,
             solvent=False, hydrogens=False, reaction_field=False),
        # the full protein-ligand setup: solvent with a cutoff and constrained hydrogens on the ligand
        dict(name="ligand_h_solvent_r1024", kind="ligand", n=2000, R=1024, k=100, precision=MIXED, check=False,
             solvent=True, hydrogens=True, reaction_field=False),
        # forward and backward: a segment and its gradient with respect to the force field and the start
        dict(name="chain22_adjoint_r256", kind="adjoint", n=22, R=256, k=200, ck=100, precision=MIXED),
        # scoring of configurations for a fit: energies, position and parameter gradients
        dict(name="chain100_energy_grad_b2048", kind="energy", n=100, B=2048, precision=MIXED),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["well", "alkanes", "chain", "chain", "chain", "chain_h", "solvated", "ions", "chains",
                       "ligand", "ligand", "adjoint", "energy"])
    prec = rng.choice([MIXED, MIXED, FP64])
    k = _log_int(rng, 50, 500)
    check = rng.random() < 0.6
    if kind == "well":
        return dict(kind=kind, R=_log_int(rng, 8, 4096), k=k)
    if kind == "alkanes":
        return dict(kind=kind, n=rng.randint(4, 7), runs=_log_int(rng, 4, 96), R=_log_int(rng, 8, 64),
                    k=_log_int(rng, 50, 200), precision=prec)
    if kind == "chain":
        n = _log_int(rng, 10, 400)
        if n >= 64 and prec == FP64:  # tiles on the FP64 path: about twenty times the mixed path's time
            return dict(kind=kind, n=n, R=_log_int(rng, 16, 128), k=_log_int(rng, 20, 50), precision=prec, check=check)
        return dict(kind=kind, n=n, R=_log_int(rng, 16, 1024 if n < 64 else 512), k=k, precision=prec, check=check)
    if kind == "chain_h":
        return dict(kind=kind, n=rng.randint(8, 31), R=_log_int(rng, 16, 512), k=_log_int(rng, 50, 200), precision=prec,
                    check=check)
    if kind == "solvated":
        return dict(kind=kind, n=_log_int(rng, 10, 63), R=_log_int(rng, 16, 512), k=k, precision=prec, check=check)
    if kind == "ions":
        if rng.random() < 0.5:  # fewer than 64 atoms: explicit pairs
            return dict(kind=kind, n=rng.randint(12, 23), pairs=rng.randint(8, 20), edge=2.6, R=_log_int(rng, 16, 512),
                        k=_log_int(rng, 50, 200), precision=MIXED, check=check)
        return dict(kind=kind, n=_log_int(rng, 40, 120), pairs=rng.randint(20, 60), edge=4.0, R=_log_int(rng, 16, 512),
                    k=_log_int(rng, 50, 200), precision=MIXED, check=check)
    if kind == "chains":
        lo = _log_int(rng, 10, 80)
        return dict(kind=kind, runs=_log_int(rng, 4, 48), R=_log_int(rng, 16, 128), lo=lo, hi=rng.randint(lo, 400),
                    k=_log_int(rng, 50, 250), precision=MIXED)
    if kind == "ligand":
        solvent, hydrogens = rng.random() < 0.4, rng.random() < 0.3
        n = 2000 if hydrogens else rng.randint(500, 2100)
        return dict(kind=kind, n=n, R=_log_int(rng, 32, 768), k=_log_int(rng, 20, 60), precision=MIXED, check=check,
                    solvent=solvent, hydrogens=hydrogens, reaction_field=not (solvent or hydrogens) and rng.random() < 0.4)
    if kind == "adjoint":
        return dict(kind=kind, n=rng.randint(10, 40), R=_log_int(rng, 16, 256), k=_log_int(rng, 50, 300),
                    ck=rng.choice([25, 50]), precision=prec)
    return dict(kind="energy", n=_log_int(rng, 10, 400), B=_log_int(rng, 64, 1024), precision=prec)


# ------------------------------------------------------------------------------------------------ systems
@functools.lru_cache(maxsize=256)
def _chain(n, seed=1807):
    return W.chain(n, seed=seed)


@functools.lru_cache(maxsize=8)
def _ligand(n, hydrogens):
    return W.ligand_receptor_h() if hydrogens else W.ligand_receptor(n_receptor=n)


def _system(case):
    """The system of a case of one system, and the state whose exits are tested."""
    kind = case["kind"]
    if kind == "well":
        return W.double_well_2d(n_replicas=case["R"]), 0
    if kind == "alkanes":
        return W.alkane(n_atoms=case["n"]), (3 ** (case["n"] - 3) - 1) // 2  # all trans
    if kind == "chain_h":
        return W.chain_h(case["n"]), 1
    if kind == "solvated":
        return W.solvated(_chain(case["n"])), 1
    if kind == "ions":
        return W.chain_ions(n_chain=case["n"], n_pairs=case["pairs"], edge=case["edge"]), 1
    if kind == "adjoint":
        return W.chain_gradient(case["n"]), 1
    if kind == "ligand":
        s = _ligand(case["n"], case["hydrogens"])
        if case["solvent"]:
            s = W.solvated(s)
        if case["reaction_field"]:
            s = dataclasses.replace(s, coulomb_mode=W.COULOMB_REACTION_FIELD)
        return s, 0
    return _chain(case["n"]), 1


def _chains(case):
    sizes = W.batched_sizes(case["runs"], 1807, case["lo"], case["hi"])
    return [_chain(int(n), 1807 + i) for i, n in enumerate(sizes)]


def _batch_systems(case):
    if case["kind"] == "chains":
        return _chains(case), [1] * case["runs"]
    s, omega = _system(case)
    return [s] * case["runs"], [omega] * case["runs"]


def _precision(case):
    return B.GRP_FP64 if case["kind"] == "well" or case["precision"] == FP64 else B.GRP_MIXED


def _start(s, R, seed):
    """Replica states of an ensemble around the system's configuration, thermal momenta."""
    return W.replica_states(s, R, seed=seed, spread=0.15 if s.potential == W.POT_DOUBLE_WELL_2D else 0.002)


def _seed(seed, i=0):
    return 2431 + 1009 * seed + i


# ------------------------------------------------------------------------------------------------ passes
def prepare(case, seed):
    B.load()
    kind = case["kind"]
    if kind in ("alkanes", "chains"):
        systems, omegas = _batch_systems(case)
        handles, reps = {}, []
        for i, s in enumerate(systems):
            if id(s) not in handles:
                handles[id(s)] = B.grp_create_system(s, _precision(case))
            q, p = _start(s, case["R"], _seed(seed, i))
            reps.append(B.grp_init_replicas(handles[id(s)], case["R"], _seed(seed, i), q, p, per_replica=True))
        batch = B.grp_batch_create(reps)
        if kind == "chains":  # uneven sizes: the program lets the library choose the block size once
            before = [B.grp_get_state(r) for r in reps]
            B.grp_batch_autotune(batch, 10)
            for r, (q, p, acc, ctr) in zip(reps, before):
                B.grp_set_state(r, q, p, acc, ctr)
        views = [B.device_tensors(r) for r in reps]
        return dict(case=case, batch=batch, omegas=np.array(omegas, np.int32), views=views, s=systems[0])
    s, omega = _system(case)
    sysh = B.grp_create_system(s, _precision(case))
    if kind == "energy":
        q, _ = _start(s, case["B"], _seed(seed))
        n_theta = B.grp_param_count(sysh)
        dev = dict(dtype=torch.float64, device="cuda")
        return dict(case=case, sysh=sysh, q=torch.from_numpy(q).cuda(), w=torch.from_numpy(_weights(case, seed)).cuda(),
                    energy=torch.empty(case["B"], **dev), grad_q=torch.empty(case["B"], s.n_atoms, 3, **dev),
                    grad_theta=torch.empty(n_theta, **dev))
    q, p = _start(s, case["R"], _seed(seed))
    rep = B.grp_init_replicas(sysh, case["R"], _seed(seed), q, p, per_replica=True)
    state = dict(case=case, s=s, omega=omega, sysh=sysh, rep=rep, views=B.device_tensors(rep), status=B.FvStatus())
    if kind == "adjoint":
        dev = dict(dtype=torch.float64, device="cuda")
        state.update(grad_theta=torch.empty(B.grp_param_count(sysh), **dev),
                     grad_q0=torch.empty(case["R"], s.n_atoms, 3, **dev),
                     grad_p0=torch.empty(case["R"], s.n_atoms, 3, **dev))
    return state


def _weights(case, seed):
    return np.random.default_rng(_seed(seed, 7)).uniform(0.5, 1.5, case["B"])


def _status(st, n_obs):
    return {"ref_exited": st.ref_exited, "label0": st.label0, "n_branched": st.n_branched,
            "converged": st.converged, "rhat": np.array(st.rhat[:n_obs])}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("alkanes", "chains"):
        s = state["s"]
        st = B.grp_batch_fv_check(state["batch"], state["omegas"], case["k"], s.t_gr, s.tol)
        out = {key: torch.cat([v[key].reshape(-1) for v in state["views"]]) for key in ("q", "p", "f", "acc")}
        n_obs = len(s.observables)
        out["rhat"] = np.array([x.rhat[:n_obs] for x in st])
        out["status"] = np.array([(x.ref_exited, x.label0, x.n_branched, x.converged) for x in st])
        return out
    if kind == "energy":
        B.grp_energy_grad(state["sysh"], case["B"], state["q"], state["w"], state["energy"], state["grad_q"],
                          state["grad_theta"])
        return {key: state[key] for key in ("energy", "grad_q", "grad_theta")}
    v, s = state["views"], state["s"]
    if kind == "adjoint":
        loss = B.grp_adjoint_segment(state["rep"], case["k"], s.t_gr, case["ck"], 4, d_grad_theta=state["grad_theta"],
                                     d_grad_q0=state["grad_q0"], d_grad_p0=state["grad_p0"])
        return {"loss": loss, "grad_theta": state["grad_theta"], "grad_q0": state["grad_q0"],
                "grad_p0": state["grad_p0"], "q": v["q"], "p": v["p"]}
    if case.get("check", True):
        st = B.grp_fv_check(state["rep"], state["omega"], case["k"], _t_gr(case, s), s.tol, 0, None, state["status"])
        return {"q": v["q"], "p": v["p"], "f": v["f"], "acc": v["acc"], "labels": v["labels"], "exited": v["exited"],
                **_status(st, len(s.observables))}
    B.grp_step_k(state["rep"], case["k"], _t_gr(case, s))
    return {"q": v["q"], "p": v["p"], "f": v["f"], "acc": v["acc"]}


def _t_gr(case, s):
    return s.t_gr if case["k"] >= s.t_gr else 10


# ------------------------------------------------------------------------------------------------ work
def _terms(s):
    """Flops of one force evaluation: 40 per pair (within the cutoff of the first configuration, where there is
    one), 15 per bond, 40 per angle, 33 per dihedral term; in solvent 110 more per pair and 20 per excluded pair;
    on the mesh a real transform forth and back, spreading and gathering; 30 per atom for the integrator."""
    if s.potential == W.POT_DOUBLE_WELL_2D:
        return 60.0
    n = s.n_atoms
    if s.cutoff > 0:
        d = s.q0[:, None] - s.q0[None]
        if s.box is not None:
            d -= np.asarray(s.box) * np.round(d / np.asarray(s.box))
        near = np.triu((d ** 2).sum(-1) < s.cutoff ** 2, 1)
        all_near = int(near.sum())
        near[s.excl[:, 0], s.excl[:, 1]] = False
        near[s.excl[:, 1], s.excl[:, 0]] = False
        pairs = int(near.sum())
    else:
        all_near = n * (n - 1) // 2
        pairs = all_near - len({tuple(sorted(e)) for e in np.asarray(s.excl).tolist()})
    f = 40.0 * pairs + 15.0 * len(s.bonds) + 40.0 * len(s.angles) + 33.3 * len(s.dihedral_k) + 30.0 * n
    if s.gb_radius is not None:
        f += 110.0 * all_near
    if s.box is not None:
        G = float(np.prod(s.pme_grid))
        f += 6.0 * pairs + 20.0 * len(s.excl) + 5.0 * G * math.log2(G) + 2.0 * G + 700.0 * n
    return f


@functools.lru_cache(maxsize=64)
def _work(items):
    case = dict(items)
    kind = case["kind"]
    if kind in ("alkanes", "chains"):
        systems, _ = _batch_systems(case)
        flops = {id(s): _terms(s) for s in systems}
        row = sum(16.0 * (3 * s.n_atoms * s.dim + 4 * len(s.observables)) for s in systems)
        return {"bytes": case["R"] * row, "flops": case["R"] * case["k"] * sum(flops[id(s)] for s in systems)}
    s, _ = _system(case)
    nd = s.n_atoms * s.dim
    if kind == "energy":
        nt = 2 * s.n_atoms + len(s.dihedral_k)
        return {"bytes": 8.0 * (case["B"] * (2 * nd + 2) + nt), "flops": case["B"] * 2.0 * _terms(s)}
    R, k = case["R"], case["k"]
    if kind == "adjoint":  # the segment, and a pass and a tangent pass per configuration on the way back
        nt = 2 * s.n_atoms + len(s.dihedral_k)
        return {"bytes": 8.0 * (R * 8 * nd + nt), "flops": 4.0 * R * k * _terms(s)}
    return {"bytes": 16.0 * R * (3 * nd + 4 * len(s.observables)), "flops": R * float(k) * _terms(s)}


def work(case):
    return dict(_work(tuple(sorted((k, v) for k, v in case.items() if k != "name"))))


# ------------------------------------------------------------------------------------------------ exact
def _philox(c, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words: counter words c[0..3], key words key[0..1]."""
    M32 = 0xFFFFFFFF

    def mul(a, b):  # high and low words of a 32 x 32-bit product; a is a number
        lo, hi = a * (b & 0xFFFF), a * (b >> 16)
        return ((hi + (lo >> 16)) >> 16) & M32, (((hi & 0xFFFF) << 16) + lo) & M32

    c0, c1, c2, c3 = c
    k0, k1 = key
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


class _Noise:
    """The normals of every step, replica and atom: [R][n][dim]."""

    def __init__(self, seeds, reps, n, dim):
        seeds = torch.as_tensor([[s & 0xFFFFFFFF, s >> 32] for s in seeds], dtype=torch.int64, device="cuda")
        self.key = seeds[:, 0, None].expand(-1, n), seeds[:, 1, None].expand(-1, n)
        self.r = torch.as_tensor(reps, dtype=torch.int64, device="cuda")[:, None].expand(-1, n)
        self.a = torch.arange(n, device="cuda").expand(len(reps), -1)
        self.dim = dim

    def words(self, t, stream):
        c0 = torch.full_like(self.r, t & 0xFFFFFFFF)
        return _philox((c0, torch.full_like(c0, ((t >> 32) & 0xFFFFFF) | (stream << 24)), self.r, self.a), self.key)

    def __call__(self, t):
        w = [(x.double() + 0.5) * 2.0 ** -32 for x in self.words(t, 0)]
        out = []
        for u1, u2 in ((w[0], w[1]), (w[2], w[3])):
            rad, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
            out += [rad * torch.cos(ang), rad * torch.sin(ang)]
        return torch.stack(out[:self.dim], -1)


def _dihedral(q, i, j, k, l):
    b1, b2, b3 = q[:, j] - q[:, i], q[:, k] - q[:, j], q[:, l] - q[:, k]
    n1, n2 = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
    return torch.atan2(b2.norm(dim=-1) * (b1 * n2).sum(-1), (n1 * n2).sum(-1))


class _Model:
    """Potential energy of a system in 64 bits, batched over configurations [B][n][dim]."""

    def __init__(self, s, margin=0.4):
        self.s = s
        t = lambda x: torch.as_tensor(np.asarray(x), device="cuda")  # noqa: E731
        self.mass = t(s.mass)[:, None]
        if s.potential == W.POT_DOUBLE_WELL_2D:
            return
        n = s.n_atoms
        ex = np.zeros((n, n), bool)
        ex[s.excl[:, 0], s.excl[:, 1]] = ex[s.excl[:, 1], s.excl[:, 0]] = True
        i, j = np.triu_indices(n, 1)
        if s.cutoff > 0 and s.box is None and n > 256:  # pairs that can come within the cutoff
            near = np.linalg.norm(s.q0[i] - s.q0[j], axis=1) < s.cutoff + margin
            i, j = i[near], j[near]
        keep = ~ex[i, j]
        self.i, self.j = t(i[keep]), t(j[keep])
        self.ai, self.aj = t(i), t(j)            # every pair, for the solvent
        self.xi, self.xj = t(i[~keep]), t(j[~keep])
        self.sigma, self.eps, self.charge = t(s.sigma), t(s.epsilon), t(s.charge)
        self.bonds, self.angles, self.dih = t(s.bonds).long(), t(s.angles).long(), t(s.dihedrals).long()
        self.bk, self.br = t(s.bond_k), t(s.bond_r0)
        self.ak, self.at = t(s.angle_k), t(s.angle_theta0)
        self.dn, self.dk, self.dd = t(s.dihedral_n).double(), t(s.dihedral_k), t(s.dihedral_delta)
        if s.gb_radius is not None:
            self.rho, self.scale = t(s.gb_radius), t(s.gb_scale)
        self.theta = [self.sigma, self.eps, self.dk]
        if s.box is not None:
            self._mesh()

    def size(self):
        return len(self.ai) if self.s.potential == W.POT_FORCE_FIELD else 1

    def _diff(self, q, i, j):
        d = q[:, i] - q[:, j]
        if self.s.box is not None:
            box = torch.tensor(self.s.box, dtype=torch.float64, device="cuda")
            d = d - box * torch.round(d.detach() / box)
        return d

    def energy(self, q, theta=None):
        s = self.s
        if s.potential == W.POT_DOUBLE_WELL_2D:
            x, y = q[:, 0, 0], q[:, 0, 1]
            return s.dw_a * (x * x - 1.0) ** 2 + s.dw_b * y * y
        sigma, eps, dk = theta if theta is not None else self.theta
        d = self._diff(q, self.i, self.j)
        r2 = (d * d).sum(-1)
        qq = s.coulomb_k / 4.0 * self.charge[self.i] * self.charge[self.j]
        s6 = (0.25 * (sigma[self.i] + sigma[self.j]) ** 2 / r2) ** 3
        e = 4.0 * torch.sqrt(eps[self.i] * eps[self.j]) * (s6 * s6 - s6)
        if s.coulomb_mode == W.COULOMB_EPS4R:
            e = e + qq / r2
        elif s.coulomb_mode == W.COULOMB_REACTION_FIELD:
            rc, er = s.cutoff, s.rf_dielectric
            krf = (0.5 if er == 0 else (er - 1.0) / (2.0 * er + 1.0)) / rc ** 3
            e = e + 4.0 * qq * (1.0 / torch.sqrt(r2) + krf * r2 - (1.0 / rc + krf * rc * rc))
        else:
            r = torch.sqrt(r2)
            e = e + 4.0 * qq * torch.erfc(s.ewald_beta * r) / r
        if s.cutoff > 0:
            e = torch.where(r2 < s.cutoff ** 2, e, torch.zeros_like(e))
        e = e.sum(-1)
        if len(self.bonds):
            r = (q[:, self.bonds[:, 0]] - q[:, self.bonds[:, 1]]).norm(dim=-1)
            e = e + (0.5 * self.bk * (r - self.br) ** 2).sum(-1)
        if len(self.angles):
            u, v = q[:, self.angles[:, 0]] - q[:, self.angles[:, 1]], q[:, self.angles[:, 2]] - q[:, self.angles[:, 1]]
            th = torch.atan2(torch.linalg.cross(u, v).norm(dim=-1), (u * v).sum(-1))
            e = e + (0.5 * self.ak * (th - self.at) ** 2).sum(-1)
        if len(self.dih):
            phi = _dihedral(q, *self.dih.T)
            e = e + (dk * (1.0 + torch.cos(self.dn * phi - self.dd))).sum(-1)
        if s.gb_radius is not None:
            e = e + self._solvent(q)
        if s.box is not None:
            e = e + self._reciprocal(q)
        return e

    def _solvent(self, q):
        s = self.s
        i, j = self.ai, self.aj
        r2 = ((q[:, i] - q[:, j]) ** 2).sum(-1)
        r = torch.sqrt(r2)
        on = r2 < s.cutoff ** 2 if s.cutoff > 0 else torch.ones_like(r2, dtype=torch.bool)
        a = self.rho - 0.009
        sp = self.scale * a

        def descreen(ai, sj):
            U, diff = r + sj, r - sj
            L = torch.maximum(ai.expand_as(r), diff.abs())
            h = (1 / L - 1 / U + 0.25 * r * (1 / U ** 2 - 1 / L ** 2) + 0.5 / r * torch.log(L / U)
                 + 0.25 * sj ** 2 / r * (1 / L ** 2 - 1 / U ** 2))
            h = h + torch.where(ai < sj - r, 2.0 * (1 / ai - 1 / L), torch.zeros_like(h))
            return torch.where(on & (ai < U), h, torch.zeros_like(h))

        total = torch.zeros(q.shape[0], s.n_atoms, dtype=torch.float64, device="cuda")
        total = total.index_add(1, i, descreen(a[i], sp[j])).index_add(1, j, descreen(a[j], sp[i]))
        psi = 0.5 * a * total
        born = 1.0 / (1.0 / a - torch.tanh(psi - 0.8 * psi ** 2 + 4.85 * psi ** 3) / self.rho)
        tau = s.coulomb_k * (1.0 / s.gb_solute_dielectric - 1.0 / s.gb_solvent_dielectric)
        bb = born[:, i] * born[:, j]
        f = torch.sqrt(r2 + bb * torch.exp(-r2 / (4.0 * bb)))
        pair = torch.where(on, self.charge[i] * self.charge[j] / f, torch.zeros_like(f))
        return -tau * pair.sum(-1) - 0.5 * tau * (self.charge ** 2 / born).sum(-1)

    def _mesh(self):
        s = self.s
        K, box = s.pme_grid, np.asarray(s.box)
        spline = np.array([1.0, 4.0, 1.0]) / 6.0  # M_4 at 1, 2, 3
        b, m = [], []
        for x in range(3):
            a = np.exp(2j * math.pi * np.outer(np.arange(K[x]), np.arange(3)) / K[x]) @ spline
            b.append(1.0 / np.abs(a) ** 2)
            m.append(np.where(np.arange(K[x]) <= K[x] // 2, np.arange(K[x]), np.arange(K[x]) - K[x]) / box[x])
        m2 = m[0][:, None, None] ** 2 + m[1][None, :, None] ** 2 + m[2][None, None] ** 2
        bm = b[0][:, None, None] * b[1][None, :, None] * b[2][None, None]
        V = box.prod()
        with np.errstate(divide="ignore", invalid="ignore"):
            G = s.coulomb_k * bm * np.exp(-(math.pi / s.ewald_beta) ** 2 * m2) / (math.pi * V * m2)
        G[0, 0, 0] = 0.0
        self.G = torch.as_tensor(G, device="cuda")
        qt, q2 = s.charge.sum(), (s.charge ** 2).sum()
        self.e_const = (-s.coulomb_k * s.ewald_beta / math.sqrt(math.pi) * q2
                        - s.coulomb_k * math.pi * qt ** 2 / (2.0 * V * s.ewald_beta ** 2))

    def _reciprocal(self, q):
        s = self.s
        K = torch.tensor(s.pme_grid, device="cuda")
        u = q / torch.tensor(s.box, dtype=torch.float64, device="cuda")
        u = (u - torch.floor(u.detach())) * K
        cell = torch.floor(u.detach())
        w = u - cell
        cell = cell.long()
        m = torch.stack([w ** 3, 4 - 6 * (1 - w) ** 2 + 3 * (1 - w) ** 3, 4 - 6 * w ** 2 + 3 * w ** 3, (1 - w) ** 3], -1) / 6
        g = (cell[..., None] - torch.arange(4, device="cuda")) % K[:, None]     # [B][n][axis][4]
        flat = ((g[:, :, 0, :, None, None] * K[1] + g[:, :, 1, None, :, None]) * K[2] + g[:, :, 2, None, None, :])
        val = self.charge[:, None, None, None] * (m[:, :, 0, :, None, None] * m[:, :, 1, None, :, None]
                                                  * m[:, :, 2, None, None, :])
        nb, size = q.shape[0], int(np.prod(s.pme_grid))
        grid = torch.zeros(nb, size, dtype=torch.float64, device="cuda").scatter_add(1, flat.reshape(nb, -1),
                                                                                    val.reshape(nb, -1))
        F = torch.fft.fftn(grid.reshape(nb, *s.pme_grid), dim=(1, 2, 3))
        e = 0.5 * (self.G * (F.real ** 2 + F.imag ** 2)).sum((1, 2, 3)) + self.e_const
        if len(self.xi):
            r = self._diff(q, self.xi, self.xj).norm(dim=-1)
            e = e - (s.coulomb_k * self.charge[self.xi] * self.charge[self.xj] * torch.erf(s.ewald_beta * r) / r).sum(-1)
        return e

    def forces(self, q):
        out = []
        step = max(1, int(1.5e7 // self.size()))
        for c in torch.split(q.detach(), step):
            c = c.requires_grad_(True)
            e = self.energy(c)
            out.append((-torch.autograd.grad(e.sum(), c)[0], e.detach()))
        return torch.cat([f for f, _ in out]), torch.cat([e for _, e in out])

    def observable(self, j, q, p, v):
        s = self.s
        kind, a = s.observables[j]
        if kind == W.OBS_POTENTIAL:
            return v
        if kind == W.OBS_KINETIC:
            return (0.5 * p * p / self.mass).sum((1, 2))
        if kind == W.OBS_COORD:
            return q[:, a[0], a[1]]
        if kind == W.OBS_DIHEDRAL:
            return _dihedral(q, *a)
        if kind == W.OBS_GROUP_DISTANCE:
            return (self._com(q, a[0]) - self._com(q, a[1])).norm(dim=-1)
        g = list(s.groups[a[0]])
        return torch.sqrt(((p[:, g] / self.mass[g]) ** 2).sum((1, 2)) / len(g))

    def _com(self, q, g):
        g = list(self.s.groups[g])
        return (q[:, g] * self.mass[g]).sum(1) / self.mass[g].sum()

    def exited(self, q, omega):
        s = self.s
        if s.cv_kind == W.CV_DOUBLE_WELL:
            return q[:, 0, 0] >= 0 if omega == 0 else q[:, 0, 0] < 0
        if s.cv_kind == W.CV_ROTAMERS:
            out = torch.zeros(len(q), dtype=torch.bool, device="cuda")
            for t in range(int(s.cv_params[0])):
                phi = torch.rad2deg(_dihedral(q, *s.cv_atoms[t:t + 4]))
                well = torch.where((phi >= 0) & (phi < 120), 0, torch.where((phi >= -120) & (phi < 0), 2, 1))
                out |= well != (omega // 3 ** t) % 3
            return out
        if s.cv_kind == W.CV_DIHEDRAL_RECT:
            a, b = (torch.rad2deg(_dihedral(q, *s.cv_atoms[t:t + 4])) for t in (0, 1))
            lo, hi, lo2, hi2 = s.cv_params
            label = torch.where((a >= lo) & (a <= hi) & (b >= lo2) & (b <= hi2), 0, 1)
        else:
            label = torch.where((self._com(q, 0) - self._com(q, 1)).norm(dim=-1) < s.cv_params[0], 0, 1)
        return label != omega


class _Bonds:
    """Constraints of independent pairs: SHAKE and RATTLE solved to rounding."""

    def __init__(self, s, h):
        c = torch.as_tensor(np.asarray(s.constraints), device="cuda").long()
        self.a, self.b, self.h = c[:, 0], c[:, 1], h
        m = torch.as_tensor(s.mass, device="cuda")
        self.wa, self.wb = (1.0 / m[self.a])[:, None], (1.0 / m[self.b])[:, None]
        self.d2 = torch.as_tensor(np.asarray(s.constraint_length), device="cuda") ** 2

    def rattle(self, q, p):
        r = q[:, self.a] - q[:, self.b]
        rv = (r * (p[:, self.a] * self.wa - p[:, self.b] * self.wb)).sum(-1, keepdim=True)
        mu = rv / ((self.wa + self.wb) * (r * r).sum(-1, keepdim=True))
        p = p.clone()
        p[:, self.a] -= mu * r
        p[:, self.b] += mu * r
        return p

    def drift(self, q, p, im):
        old = q[:, self.a] - q[:, self.b]
        q, p = q + self.h * p * im, p.clone()
        r = q[:, self.a] - q[:, self.b]
        w = (self.wa + self.wb)[:, 0]
        A, Bh, C = w * w * (old * old).sum(-1), w * (old * r).sum(-1), (r * r).sum(-1) - self.d2
        g = (-C / (Bh + torch.sqrt(Bh * Bh - A * C)))[..., None]
        q[:, self.a] += g * self.wa * old
        q[:, self.b] -= g * self.wb * old
        p[:, self.a] += g / self.h * old
        p[:, self.b] -= g / self.h * old
        return q, self.rattle(q, p)


def _segment(model, noise, q, p, k, t_gr):
    """k BAOAB steps from (q, p) at step 0; (q, p, f, acc) after them."""
    s = model.s
    h, c1, im = 0.5 * s.dt, math.exp(-s.gamma * s.dt), 1.0 / model.mass
    sd = torch.sqrt((1.0 - c1 * c1) * s.kT * model.mass)
    bonds = _Bonds(s, h) if s.constraints is not None else None
    f, _ = model.forces(q)
    acc = torch.zeros(len(q), len(s.observables), 4, dtype=torch.float64, device="cuda")
    for t in range(k):
        p = p + h * f
        if bonds:
            q, p = bonds.drift(q, bonds.rattle(q, p), im)
            q, p = bonds.drift(q, bonds.rattle(q, c1 * p + sd * noise(t)), im)
        else:
            q = q + h * p * im
            p = c1 * p + sd * noise(t)
            q = q + h * p * im
        f, v = model.forces(q)
        p = p + h * f
        if bonds:
            p = bonds.rattle(q, p)
        if (t + 1) % t_gr == 0:
            for j in range(len(s.observables)):
                o = model.observable(j, q, p, v)
                acc[:, j, 0] = torch.where(acc[:, j, 3] == 0, o, acc[:, j, 0])
                d = o - acc[:, j, 0]
                acc[:, j, 1] += d
                acc[:, j, 2] += d * d
                acc[:, j, 3] += 1.0
    return q, p, f, acc


def _branch(exited, word):
    """Source of every replica: itself, or for an exited worker the survivor that its random word picks."""
    ex = exited.cpu().numpy()
    src = np.arange(len(ex))
    alive = [r for r in range(1, len(ex)) if not ex[r]]
    for r in range(1, len(ex)):
        if ex[r]:
            src[r] = alive[(int(word[r]) * len(alive)) >> 32] if alive else 0
    return torch.as_tensor(src, device="cuda")


def _ratios(acc):
    a = acc[1:]
    m1 = a[..., 1] / a[..., 3]
    mk = a[..., 0] + m1
    between = ((mk - mk.mean(0)) ** 2).mean(0)
    within = (a[..., 2] / a[..., 3] - m1 ** 2).mean(0)
    return 1.0 + between / within


def _cost(s, R, k):
    """Seconds of an exact segment, about."""
    pairs = s.n_atoms ** 2 / 2
    if s.cutoff > 0 and s.n_atoms > 256 and s.box is None:
        pairs = min(pairs, 75.0 * s.n_atoms)
    per = (600.0 if s.gb_radius is not None else 150.0) * pairs
    if s.box is not None:
        per += 4.0e4 * s.n_atoms + 2.0e5
    return k * max(0.006 if s.gb_radius is not None or s.box is not None else 0.004, R * per / 2.5e11)


def _exact_checks(systems, omegas, R, k, t_gr, seeds, check):
    """Runs of one system, R replicas each, as one set."""
    s = systems[0]
    model = _Model(s)
    start = [_start(s, R, sd) for sd in seeds]
    q, p = (torch.as_tensor(np.concatenate([x[c] for x in start]), device="cuda") for c in (0, 1))
    reps = list(range(R)) * len(seeds)
    noise = _Noise([sd for sd in seeds for _ in range(R)], reps, s.n_atoms, s.dim)
    q, p, f, acc = _segment(model, noise, q, p, k, t_gr)
    rhat = []
    if check:
        words = noise.words(k, 1)[0][:, 0].cpu().numpy()
        for i, omega in enumerate(omegas):
            at = slice(i * R, (i + 1) * R)
            src = _branch(model.exited(q[at], omega), words[at])
            for x in (q, p, f, acc):
                x[at] = x[at][src]
            rhat.append(_ratios(acc[at]).cpu().numpy())
    return q, p, f, acc, np.array(rhat)


def _adjoint(model, noise, q, p, k, t_gr, obs):
    """(loss, gradients with respect to theta, q0 and p0, final q and p) of a segment's mean observable."""
    s = model.s
    h, c1, im = 0.5 * s.dt, math.exp(-s.gamma * s.dt), 1.0 / model.mass
    sd = torch.sqrt((1.0 - c1 * c1) * s.kT * model.mass)
    path = []
    f, _ = model.forces(q)
    for t in range(k):
        path.append((q, p))
        p = p + h * f
        q = q + h * p * im
        p = c1 * p + sd * noise(t)
        q = q + h * p * im
        f, _ = model.forces(q)
        p = p + h * f
    end = q, p
    norm = 1.0 / (len(q) * (k // t_gr))
    theta = [x.clone().requires_grad_(True) for x in model.theta]
    gth = [torch.zeros_like(x) for x in theta]
    # back through p += h f(q); q += ...: each force is used at the end of a step and at the start of the next
    lq, lp, loss = torch.zeros_like(q), torch.zeros_like(p), 0.0

    def pull(x, cotangent):  # the force's vector-Jacobian product at x
        y = x.detach().requires_grad_(True)
        g = torch.autograd.grad(model.energy(y, theta).sum(), y, create_graph=True)[0]
        out = torch.autograd.grad(g, [y] + theta, grad_outputs=-cotangent, allow_unused=True)
        for a, b in zip(gth, out[1:]):
            if b is not None:
                a += b
        return out[0]

    nxt, lf = q, torch.zeros_like(q)  # lf: cotangent of the force at `nxt` from the step after it
    for t in range(k - 1, -1, -1):
        if (t + 1) % t_gr == 0:
            y = nxt.detach().requires_grad_(True)
            o = model.observable(obs, y, None, None)
            loss += float(o.sum()) * norm
            lq = lq + torch.autograd.grad(o.sum() * norm, y)[0]
        lq = lq + pull(nxt, lf + h * lp)
        lp = lp + h * im * lq
        lp = c1 * lp
        lp = lp + h * im * lq
        lf = h * lp
        nxt = path[t][0]
    lq = lq + pull(nxt, lf)
    return loss, torch.cat(gth), lq, lp, *end


def exact(case, seed):
    kind = case["kind"]
    if kind in ("alkanes", "chains"):
        systems, omegas = _batch_systems(case)
        same = kind == "alkanes"
        cost = (_cost(systems[0], case["R"] * case["runs"], case["k"]) if same else
                sum(_cost(s, case["R"], case["k"]) for s in systems))
        if cost > 12.0:
            return None
        seeds = [_seed(seed, i) for i in range(case["runs"])]
        t_gr = systems[0].t_gr
        if same:
            parts = [_exact_checks(systems, omegas, case["R"], case["k"], t_gr, seeds, True)]
        else:
            parts = [_exact_checks([s], [o], case["R"], case["k"], t_gr, [sd], True)
                     for s, o, sd in zip(systems, omegas, seeds)]
        out = {key: torch.cat([x[c].reshape(-1) for x in parts]) for c, key in enumerate(("q", "p", "f", "acc"))}
        return {**out, "rhat": np.concatenate([x[4] for x in parts]), "status": None}
    s, omega = _system(case)
    if kind == "energy":
        model = _Model(s)
        q, w = torch.as_tensor(_start(s, case["B"], _seed(seed))[0], device="cuda"), _weights(case, seed)
        theta = [x.clone().requires_grad_(True) for x in model.theta]
        es, gq, gth = [], [], [torch.zeros_like(x) for x in theta]
        step = max(1, int(1.5e7 // model.size()))
        for c, cw in zip(torch.split(q, step), torch.split(torch.as_tensor(w, device="cuda"), step)):
            c = c.clone().requires_grad_(True)
            e = model.energy(c, theta)
            g = torch.autograd.grad((e * cw).sum(), [c] + theta)
            es.append(e.detach())
            gq.append(g[0])
            gth = [a + b for a, b in zip(gth, g[1:])]
        return {"energy": torch.cat(es), "grad_q": torch.cat(gq), "grad_theta": torch.cat(gth)}
    R, k = case["R"], case["k"]
    if _cost(s, R, k) * (5.0 if kind == "adjoint" else 1.0) > 12.0:
        return None
    if kind == "adjoint":
        model = _Model(s)
        q, p = (torch.as_tensor(x, device="cuda") for x in _start(s, R, _seed(seed)))
        noise = _Noise([_seed(seed)] * R, list(range(R)), s.n_atoms, s.dim)
        loss, gth, gq, gp, q, p = _adjoint(model, noise, q, p, k, s.t_gr, 4)
        return {"loss": loss, "grad_theta": gth, "grad_q0": gq, "grad_p0": gp, "q": q, "p": p}
    check = case.get("check", True)
    q, p, f, acc, rhat = _exact_checks([s], [omega], R, k, _t_gr(case, s), [_seed(seed)], check)
    out = {"q": q, "p": p, "f": f, "acc": acc}
    if check:
        out.update(labels=None, exited=None, ref_exited=None, label0=None, n_branched=None, converged=None, rhat=rhat[0])
    return out
