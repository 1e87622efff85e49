"""Kernels whose launch shape follows the number of replicas: the double well's groups of replicas per block, and
the block sizes of item-table systems, single and batched, against the FP64 oracle or a set of another size."""
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
