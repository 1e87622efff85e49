"""Kernels whose launch shape follows the number of replicas: the double well's groups of replicas per block, and
the block sizes of item-table systems, single and batched, against the FP64 oracle or a set of another size."""
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


@pytest.fixture(scope="module")
def oracle_mod():
    import oracle

    oracle.build()
    return oracle


@pytest.mark.parametrize("R", [1, 3, 1216, 1217, 1219, 4864, 4865, 4879])
@pytest.mark.parametrize("k", [1, 130])
def test_double_well_groups(B, oracle_mod, R, k):
    """k steps of R replicas against the oracle on replicas from both ends of the set: FP64 on both sides, so they
    differ by the rounding of their logarithms and sines (1e-12 is ten times what 130 steps of it give) and
    by nothing else."""
    s = W.double_well_2d(n_replicas=R)
    q0, p0 = W.replica_states(s, R, seed=3, spread=0.2)
    rep = B.grp_init_replicas(B.grp_create_system(s, B.GRP_FP64), R, SEED, q0, p0, per_replica=True)
    B.grp_step_k(rep, k, 5)
    q, p, acc, _ = B.grp_get_state(rep)
    for lo in {0, max(0, R - 20)}:
        hi = min(R, lo + 20)
        o = oracle_mod.Oracle(s)
        qo, po = q0[:hi].copy(), p0[:hi].copy()
        fo = np.stack([o.forces(qo[r]) for r in range(hi)])
        # the oracle numbers its replicas from 0: run up to hi and compare [lo, hi)
        if hi > 200:
            continue
        samples = o.step_k(qo, po, fo, SEED, 0, 0, k, 5, cap=max(1, k // 5))
        assert np.abs(q[lo:hi] - qo[lo:hi]).max() < 1e-12 and np.abs(p[lo:hi] - po[lo:hi]).max() < 1e-12
    if R > 200:  # the upper end: the same replicas as the shard that starts there, in a small set
        lo = R - 7
        part = B.grp_init_replicas(B.grp_create_system(s, B.GRP_FP64), 7, SEED, q0[lo:], p0[lo:], per_replica=True)
        B.grp_set_shard(part, lo, R)
        B.grp_step_k(part, k, 5)
        qs, ps, accs, _ = B.grp_get_state(part)
        assert np.array_equal(q[lo:], qs) and np.array_equal(p[lo:], ps) and np.array_equal(acc[lo:], accs)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("make", ["chain10", "chain22", "chain40", "chain_h", "solvated"])
def test_block_sizes_give_the_same_bits(B, make, prec):
    """Large sets run with smaller blocks than small ones: the fixed-point sums do not depend on the
    decomposition, so the first replicas are those of a small set bit for bit."""
    s = {"chain10": lambda: W.chain(10), "chain22": lambda: W.chain(22), "chain40": lambda: W.chain(40),
         "chain_h": lambda: W.chain_h(12), "solvated": lambda: W.solvated(W.chain(14))}[make]()
    R, small, k = 2600, 5, 12
    q0, p0 = W.replica_states(s, R, seed=9, spread=0.002)
    sysh = B.grp_create_system(s, B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED)
    out = []
    for n in (small, 320, 470, R):
        rep = B.grp_init_replicas(sysh, n, SEED, q0[:n], p0[:n], per_replica=True)
        B.grp_step_k(rep, k, 4)
        q, p, acc, _ = B.grp_get_state(rep)
        out.append((q[:small], p[:small], acc[:small]))
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n_runs", [2, 40, 130])
def test_batched_block_sizes_give_the_same_bits(B, n_runs):
    """Batches of small systems: up to 130 x 20 = 2,600 units, against the runs alone."""
    s, R, k = W.alkane(), 20, 30
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    q0, p0 = W.replica_states(s, R, seed=2, spread=0.002)
    runs = [B.grp_init_replicas(sysh, R, SEED + i, q0, p0, per_replica=True) for i in range(n_runs)]
    B.grp_batch_step_k(B.grp_batch_create(runs), k, 5)
    for i in (0, n_runs - 1):
        alone = B.grp_init_replicas(sysh, R, SEED + i, q0, p0, per_replica=True)
        B.grp_step_k(alone, k, 5)
        for a, b in zip(B.grp_get_state(alone)[:3], B.grp_get_state(runs[i])[:3]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("make", ["chain_h22", "chain_h30", "rf40", "cutoff40", "chain60", "solvated40"])
def test_kernel_variants_give_the_same_bits(B, make, prec):
    """Systems of more than 320 items, whose large sets run another instantiation of the kernel than the small ones: the
    first replicas are the small set's bit for bit."""
    s = {"chain_h22": lambda: W.chain_h(22), "chain_h30": lambda: W.chain_h(30),
         "rf40": lambda: dataclasses.replace(W.chain(40), cutoff=1.0, coulomb_mode=W.COULOMB_REACTION_FIELD),
         "cutoff40": lambda: dataclasses.replace(W.chain(40), cutoff=1.0), "chain60": lambda: W.chain(60),
         "solvated40": lambda: W.solvated(W.chain(40))}[make]()
    small, k = 4, 24
    q0, p0 = W.replica_states(s, 700, seed=9, spread=0.002)
    sysh = B.grp_create_system(s, B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED)
    out = []
    for n in (small, 200, 400, 700):
        rep = B.grp_init_replicas(sysh, n, SEED, q0[:n], p0[:n], per_replica=True)
        B.grp_step_k(rep, k, 4)
        out.append([x[:small] for x in B.grp_get_state(rep)[:3]])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("make", ["chain10", "chain40", "rf22", "rf40", "alkane5"])
@pytest.mark.parametrize("n_runs", [1, 100])
def test_batches_give_the_bits_of_runs_alone(B, make, prec, n_runs):
    """Batches of small systems on both precisions, with and without the reaction field: up to 400 units."""
    rf = lambda n: dataclasses.replace(W.chain(n), cutoff=1.0, coulomb_mode=W.COULOMB_REACTION_FIELD)
    s = {"chain10": lambda: W.chain(10), "chain40": lambda: W.chain(40), "rf22": lambda: rf(22), "rf40": lambda: rf(40),
         "alkane5": lambda: W.alkane(5)}[make]()
    R, k = 4, 24
    q0, p0 = W.replica_states(s, R, seed=9, spread=0.002)
    sysh = B.grp_create_system(s, B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED)
    alone, *runs = (B.grp_init_replicas(sysh, R, SEED, q0, p0, per_replica=True) for _ in range(n_runs + 1))
    B.grp_step_k(alone, k, 4)
    B.grp_batch_step_k(B.grp_batch_create(runs), k, 4)
    for r in (runs[0], runs[-1]):
        for a, b in zip(B.grp_get_state(alone)[:3], B.grp_get_state(r)[:3]):
            assert np.array_equal(a, b)


def _best_ms(step, n=5):
    import torch

    t = []
    for _ in range(n):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        step()
        e[1].record()
        torch.cuda.synchronize()
        t.append(e[0].elapsed_time(e[1]))
    return min(t)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_twice_the_replicas_take_twice_as_long(B, prec):
    """A set of two full waves takes two waves' time: twice the replicas that fill the chip in two blocks per SM take at
    most 1.15 times twice as long (in two waves of smaller blocks, the second almost empty, 1.26 times)."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = W.solvated(W.chain(60))
    sysh = B.grp_create_system(s, B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED)
    q0, p0 = W.replica_states(s, 4 * sms, seed=3, spread=0.002)
    ms = []
    for R in (2 * sms, 4 * sms):
        rep = B.grp_init_replicas(sysh, R, SEED, q0[:R], p0[:R], per_replica=True)
        ms.append(_best_ms(lambda: B.grp_step_k(rep, 10, 10)))
    assert ms[1] <= 1.15 * 2.0 * ms[0]


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("sizes", [(60, 10, 10, 10, 10, 10, 10, 10), (10, 22, 40, 60)])
def test_uneven_batches_keep_large_blocks(B, sizes, prec):
    """A few large replicas among many small ones decide a batch's time: 256 units of uneven sizes take at most 1.25 times
    as long as a batch of the largest runs alone (with blocks for 256 even units they took 1.6 times)."""
    p = B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED
    runs = []
    for i in range(8):
        s = W.chain(sizes[i % len(sizes)])
        q0, p0 = W.replica_states(s, 32, seed=i, spread=0.002)
        runs.append(B.grp_init_replicas(B.grp_create_system(s, p), 32, SEED + i, q0, p0, per_replica=True))
    largest = [r for i, r in enumerate(runs) if sizes[i % len(sizes)] == 60]
    k = 40 if prec == "mixed" else 10
    ms = [_best_ms(lambda b=B.grp_batch_create(x): B.grp_batch_step_k(b, k, 10)) for x in (largest, runs)]
    assert ms[1] <= 1.25 * ms[0]


def test_transients_of_a_batch_keep_large_blocks(B):
    """Runs in a transient advance one replica each, whatever their sets: 64 runs of 32 replicas take at most 1.25 times as
    long as 64 of 4 (with the blocks of 2,048 replicas they took 1.6 times), and see the same events."""
    s = W.alkane(core_half_width=0.01)  # hardly ever inside a state's core
    out = []
    for R in (4, 32):
        sysh = B.grp_create_system(s, B.GRP_MIXED)
        runs = []
        for i in range(64):
            q0, p0 = W.replica_states(s, R, seed=i, spread=0.002)
            q0[:], p0[:] = W.replica_states(s, 1, seed=i, spread=0.02)[0], W.replica_states(s, 1, seed=i)[1]
            runs.append(B.grp_init_replicas(sysh, R, SEED + i, q0, p0, per_replica=True))
        batch, ends = B.grp_batch_create(runs), iter(range(2000, 20000, 2000))
        out.append((_best_ms(lambda: B.grp_batch_run(batch, 10, 100, 0.05, 1000, next(ends), 100), 4),
                    [B.grp_get_state(r)[0][0] for r in runs]))
    assert out[1][0] <= 1.25 * out[0][0]
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("make,n_runs,R", [("alkane", 64, 32), ("chain22", 8, 40), ("mixed sizes", 8, 32)])
def test_autotuning_keeps_the_faster_block_size(B, make, n_runs, R):
    """A batch is no slower after its tuning than before (1.15: two timings of one size differ by less), and tuning it
    again finds the same."""
    runs = []
    for i in range(n_runs):
        s = W.alkane() if make == "alkane" else W.chain(22 if make == "chain22" else (10, 22, 40, 60)[i % 4])
        q0, p0 = W.replica_states(s, R, seed=i, spread=0.002)
        runs.append(B.grp_init_replicas(B.grp_create_system(s, B.GRP_MIXED), R, SEED + i, q0, p0, per_replica=True))
    batch = B.grp_batch_create(runs)
    ms = [_best_ms(lambda: B.grp_batch_step_k(batch, 100, 10))]
    for _ in range(2):
        assert 32 <= B.grp_batch_autotune(batch, 10) <= 512
        ms.append(_best_ms(lambda: B.grp_batch_step_k(batch, 100, 10)))
    assert max(ms[1:]) <= 1.15 * ms[0]


@pytest.mark.parametrize("per_sm", [(3, 8), (4, 8), (6, 9), (16, 32), (20, 32)])
def test_double_well_time_grows_with_replicas(B, per_sm):
    """A smaller set is no slower than a larger one (1.1: two timings of one differ by less): the number of replicas per
    block changes where the times cross.  (With one per block up to eight per SM, 913 to 1,216 replicas took 1.7 times as
    long as 1,217, and up to 32 per SM with four, 3,649 to 4,864 took 1.2 times as long as 4,865.)"""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ms = []
    for R in (per_sm[0] * sms, per_sm[0] * sms + 1, per_sm[1] * sms, per_sm[1] * sms + 1):
        s = W.double_well_2d(n_replicas=R)
        q0, p0 = W.replica_states(s, R, seed=3, spread=0.1)
        rep = B.grp_init_replicas(B.grp_create_system(s, B.GRP_FP64), R, SEED, q0, p0, per_replica=True)
        ms.append(_best_ms(lambda: B.grp_step_k(rep, 2000, 10)))
    assert all(a <= 1.1 * b for a, b in zip(ms, ms[1:]))


@pytest.mark.parametrize("R", [456, 457, 459, 2432, 2433, 2447])
def test_double_well_lines(B, R):
    """On both sides of the lines: the last replicas are those of the shard that starts there, in a small set."""
    s = W.double_well_2d(n_replicas=R)
    q0, p0 = W.replica_states(s, R, seed=3, spread=0.2)
    sysh = B.grp_create_system(s, B.GRP_FP64)
    rep = B.grp_init_replicas(sysh, R, SEED, q0, p0, per_replica=True)
    B.grp_step_k(rep, 130, 5)
    part = B.grp_init_replicas(sysh, 7, SEED, q0[R - 7:], p0[R - 7:], per_replica=True)
    B.grp_set_shard(part, R - 7, R)
    B.grp_step_k(part, 130, 5)
    for a, b in zip(B.grp_get_state(rep)[:3], B.grp_get_state(part)[:3]):
        assert np.array_equal(a[R - 7:], b)
