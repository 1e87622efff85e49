"""Host threads that use the library at the same time, each on objects of its own."""
import threading

import pytest

from paper_1807_02431_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_systems_and_batches_made_beside_running_ones():
    """One thread advances a set and a batch that need more than 48 KB of shared memory while two others make systems and
    batches of the same kernels that need less: no launch is refused."""
    from paper_1807_02431_gb300 import binding as B

    B.load()

    def replicas(s):
        q0, p0 = W.replica_states(s, 2, seed=1, spread=0.002)
        sysh = B.grp_create_system(s, B.GRP_MIXED)
        return sysh, [B.grp_init_replicas(sysh, 2, 1, q0, p0, per_replica=True) for _ in range(2)]

    _, (rep, _) = replicas(W.solvated(W.chain(60)))
    _, (_, run) = replicas(W.chain(300))
    _, (_, small) = replicas(W.chain(30))
    batch = B.grp_batch_create([run])
    errors, done = [], threading.Event()

    def make():
        s = W.solvated(W.chain(30))
        while not done.is_set():
            B.grp_create_system(s, B.GRP_MIXED)
            B.grp_batch_create([small])

    makers = [threading.Thread(target=make) for _ in range(2)]
    for m in makers:
        m.start()
    try:
        for _ in range(12000):
            B.grp_step_k(rep, 1, 0)
            B.grp_batch_step_k(batch, 1, 0)
    except B.GrpError as e:
        errors.append(e)
    finally:
        done.set()
        for m in makers:
            m.join()
    assert not errors
    B.grp_get_state(rep)
