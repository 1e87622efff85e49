"""Neighbour rows (large systems in vacuum on the mixed path) against the pair list of the batched kernel, which
keeps it: the sums are integers, so the two agree bit for bit, over sizes around the tiles and the line between the
two forms, with and without constraints and reaction field, through several rebuilds; and rows that outgrow their
pieces (a dense clump) fall back to pairs."""
import dataclasses

import numpy as np
import pytest

from paper_1807_02431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
SEED = 2431


@pytest.fixture(scope="module")
def B():
    from paper_1807_02431_gb300 import binding

    binding.load()
    return binding


def _pair(B, s, R, k, t_gr, seed=6):
    """The same replicas advanced alone (rows) and in a batch of one run (pairs)."""
    q0, p0 = W.replica_states(s, R, seed=seed, spread=0.002)
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    alone, run = (B.grp_init_replicas(sysh, R, SEED, q0, p0, per_replica=True) for _ in range(2))
    B.grp_step_k(alone, k, t_gr)
    B.grp_batch_step_k(B.grp_batch_create([run]), k, t_gr)
    return B.grp_get_state(alone)[:3], B.grp_get_state(run)[:3]


@pytest.mark.parametrize("n,rf", [(993, False), (994, False), (995, True), (1023, False), (1500, True), (1840, False),
                                  (2000, False), (2100, True)])
def test_rows_give_the_bits_of_the_pair_list(B, n, rf):
    s = W.ligand_receptor(n_receptor=n)
    if rf:
        s = dataclasses.replace(s, coulomb_mode=W.COULOMB_REACTION_FIELD)
    for a, b in zip(*_pair(B, s, 3, 120, 20)):
        assert np.array_equal(a, b)


def test_rows_with_constraints(B, oracle_mod):
    """Constrained hydrogens are not batched: one step against the FP64 oracle, with the tolerances of the other
    one-step tests of the mixed path."""
    s = W.ligand_receptor_h()
    q0, p0 = W.replica_states(s, 2, seed=4, spread=0.0)
    rep = B.grp_init_replicas(B.grp_create_system(s, B.GRP_MIXED), 2, SEED, q0, p0, per_replica=True)
    B.grp_step_k(rep, 1, 0)
    q, p = B.grp_get_state(rep)[:2]
    o = oracle_mod.Oracle(s)
    qo, po = q0.copy(), p0.copy()
    fo = np.stack([o.forces(qo[r]) for r in range(2)])
    o.step_k(qo, po, fo, SEED, 0, 0, 1, 0, cap=1)
    assert np.abs(q - qo).max() <= 1e-9 * np.abs(qo).max() and np.abs(p - po).max() <= 1e-6 * np.abs(po).max()


@pytest.fixture(scope="module")
def oracle_mod():
    import oracle

    oracle.build()
    return oracle


@pytest.mark.parametrize("side", [0, 8, 10])
def test_dense_clumps(B, side):
    """A clump of side^3 weakly charged beads on a lattice of 0.12 nm (no Lennard-Jones) in a sparse gas: up to 1,000
    partners within the cutoff, more than a row's 256 places or the pool's blocks, beside a sparse rest.  The largest
    force is some ten kJ/mol/nm."""
    n = 1100
    rng = np.random.default_rng(3)
    x = np.stack(np.meshgrid(*[np.arange(11)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * 0.9
    m = side ** 3
    if m:
        x[:m] = 20.0 + 0.12 * np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
    s = W.System(name="gas", n_atoms=n, dim=3, potential=W.POT_FORCE_FIELD, mass=np.full(n, 12.0), kT=0.1, gamma=1.0,
                 dt=0.002, sigma=np.full(n, 0.05), epsilon=np.zeros(n), charge=rng.normal(0, 0.01, n),
                 excl=np.zeros((0, 2), np.int32), cutoff=1.2, coulomb_k=W.COULOMB_K, cv_kind=W.CV_COM_DISTANCE,
                 cv_params=(1.0,), groups=[[0], [1]], observables=[(W.OBS_POTENTIAL, ()), (W.OBS_KINETIC, ())])
    s.q0, s.p0 = x, W.maxwell_boltzmann(s.mass, s.kT, 3, rng)
    for a, b in zip(*_pair(B, s, 2, 40, 10)):
        assert np.array_equal(a, b)


def _gas(n, cutoff, seed=3):
    """n weakly charged beads on a lattice of 0.9 nm."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1 / 3)))
    x = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * 0.9
    s = W.System(name="gas", n_atoms=n, dim=3, potential=W.POT_FORCE_FIELD, mass=np.full(n, 12.0), kT=0.1, gamma=1.0,
                 dt=0.002, sigma=np.full(n, 0.3), epsilon=np.full(n, 0.1), charge=rng.normal(0, 0.1, n),
                 excl=np.zeros((0, 2), np.int32), cutoff=cutoff, coulomb_k=W.COULOMB_K, cv_kind=W.CV_COM_DISTANCE,
                 cv_params=(1.0,), groups=[[0], [1]], observables=[(W.OBS_POTENTIAL, ()), (W.OBS_KINETIC, ())])
    s.q0, s.p0 = x, W.maxwell_boltzmann(s.mass, s.kT, 3, rng)
    return s


@pytest.mark.parametrize("prec,n,cutoff", [(1, 2380, 1.2), (1, 2381, 1.2), (1, 2393, 1.2), (1, 2394, 1.2), (1, 2484, 1.2),
                                           (1, 2504, 0.0), (0, 2381, 1.2), (0, 2400, 0.0)])
def test_largest_batched_systems(B, prec, n, cutoff):
    """The largest systems that a batch can hold beside its 1,120 bytes of launch arguments, on both precisions, with
    and without lists, and the sizes at which the single run's charge array stops fitting (2,393): accepted, and equal to
    the run alone."""
    s = _gas(n, cutoff)
    sysh = B.grp_create_system(s, B.GRP_MIXED if prec else B.GRP_FP64)
    alone, run = (B.grp_init_replicas(sysh, 1, SEED, s.q0[None], s.p0[None], per_replica=True) for _ in range(2))
    B.grp_step_k(alone, 3, 1)
    B.grp_batch_step_k(B.grp_batch_create([run]), 3, 1)
    for a, b in zip(B.grp_get_state(alone)[:3], B.grp_get_state(run)[:3]):
        assert np.array_equal(a, b)


def _globule(n, rho, seed=1):
    """n weakly interacting beads at rho per nm^3, numbered along the lattice."""
    rng = np.random.default_rng(seed)
    a = rho ** (-1.0 / 3.0)
    s = _gas(n, 1.2, seed)
    m = int(np.ceil(n ** (1 / 3)))
    s.q0 = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * a + rng.uniform(-0.02, 0.02, (n, 3))
    return dataclasses.replace(s, sigma=np.full(n, 0.6 * a), epsilon=np.full(n, 0.05), q0=s.q0, p0=s.p0, dt=0.001)


@pytest.mark.parametrize("n,rho", [(1100, 60), (1100, 100), (2030, 100)])
def test_dense_systems_keep_the_speed_of_pairs(B, n, rho):
    """A set whose rows would be longer than their 256 places takes the pair list: as fast as the batched kernel,
    which always does, within a third (through rows of one pair each it took three times as long)."""
    import torch

    s = _globule(n, rho)
    q0, p0 = W.replica_states(s, 8, seed=6, spread=0.0005)
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    alone, run = (B.grp_init_replicas(sysh, 8, SEED, q0, p0, per_replica=True) for _ in range(2))
    batch = B.grp_batch_create([run])
    ms = []
    for step in (lambda: B.grp_step_k(alone, 20, 10), lambda: B.grp_batch_step_k(batch, 20, 10)):
        t = []
        for _ in range(4):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            step()
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        ms.append(min(t))
    assert ms[0] <= 1.33 * ms[1]
    for a, b in zip(B.grp_get_state(alone)[:3], B.grp_get_state(run)[:3]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("hub", [400, 600])
def test_rows_outgrown_by_one_replica(B, hub):
    """Replica 0, whose configuration decides, is a sparse gas; in replica 1 `hub` beads sit on a sphere of 1.3 nm around
    one (a row of 200 partners, which fits, or of 300, which does not): that replica goes on in pairs."""
    s = _gas(1100, 1.2)
    s = dataclasses.replace(s, epsilon=np.zeros(1100), charge=s.charge * 0.1, q0=s.q0, p0=s.p0)
    q1 = s.q0.copy() + 20.0
    z = (2.0 * np.arange(hub) + 1.0) / hub - 1.0  # evenly: equal bands, the golden angle apart
    phi = np.arange(hub) * np.pi * (3.0 - np.sqrt(5.0))
    q1[0] = 0.0
    q1[1:hub + 1] = 1.3 * np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], -1)
    d = np.linalg.norm(q1[:, None] - q1[None], axis=-1) < 1.4
    row0 = sum(d[0, j] for j in range(1, 1100) if j % 2)
    assert (row0 > 256) == (hub > 512) and np.triu(d, 1).sum() < 65536
    q0, p0 = np.stack([s.q0, q1, s.q0]), np.stack([s.p0] * 3)
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    alone, run = (B.grp_init_replicas(sysh, 3, SEED, q0, p0, per_replica=True) for _ in range(2))
    for k in (1, 40):
        B.grp_step_k(alone, k, 10)
        B.grp_batch_step_k(B.grp_batch_create([run]), k, 10)
        for a, b in zip(B.grp_get_state(alone)[:3], B.grp_get_state(run)[:3]):
            assert np.array_equal(a, b)


def test_systems_with_rows_are_made_quickly(B):
    """The rows' tables add at most a third to the time in which a system is made: one of 1,024 atoms against one of 1,022,
    which has none (they more than doubled it)."""
    import time

    def best(n):
        s = _gas(n, 1.2)
        t = []
        for _ in range(7):
            t0 = time.perf_counter()
            B.grp_create_system(s, B.GRP_MIXED)
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(1024) <= 1.33 * best(1022)
