"""The integer conversions to the 2^-40 fixed point, through the forces of one bond whose arithmetic is
exact, and the column sums of the parameter gradient at the edges of their row blocks."""
import numpy as np
import pytest

from paper_1807_02431_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_1807_02431_gb300 import binding

    binding.load()
    return binding


def _bond(k, x, r0):
    """Two atoms x apart on the first axis, one bond (k, r0) and nothing else."""
    s = W.System(name="bond", n_atoms=2, dim=3, potential=W.POT_FORCE_FIELD, mass=np.ones(2), kT=1.0, gamma=1.0, dt=1e-3,
                 sigma=np.full(2, 0.3), epsilon=np.zeros(2), charge=np.zeros(2), excl=np.array([[0, 1]], np.int32),
                 bonds=np.array([[0, 1]], np.int32), bond_k=np.array([k]), bond_r0=np.array([r0]),
                 cv_kind=W.CV_COM_DISTANCE, cv_params=(1.0,), groups=[[0], [1]])
    s.q0, s.p0 = np.array([[0.0, 0, 0], [x, 0, 0]]), np.zeros((2, 3))
    return s


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("e", [-60, -43, -42, -41, -40, -39, -30, -20, -10, 0, 11, 12, 13, 20, 21])
def test_fp64_fixed_point_of_a_force(B, e, sign):
    """Force k (r - r0) with every factor a few bits long, so that it is exact before the conversion: the
    result is the nearest multiple of 2^-40 (ties to even), whatever its size below 2^22."""
    import torch

    for m in (1.0, 1.5, 1.25, 1.75, 1.0 + 2.0 ** -12):
        x, r0 = (2.0, 1.0) if sign > 0 else (1.0, 2.0)
        k = m * 2.0 ** e  # force on atom 0 towards atom 1 when stretched: k (r - r0) = +-k
        sysh = B.grp_create_system(_bond(k, x, r0), B.GRP_FP64)
        q = torch.tensor([[[0.0, 0, 0], [x, 0, 0]]], dtype=torch.float64, device="cuda")
        f = torch.empty_like(q)
        B.grp_energy_forces(sysh, 1, q, None, f)
        want = sign * np.rint(k * 2.0 ** 40) * 2.0 ** -40
        assert f[0, 0, 0].item() == want and f[0, 1, 0].item() == -want


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n_conf", [1, 2, 63, 64, 65, 127, 129, 200])
def test_param_gradient_sums(B, n_conf, prec):
    """The summed parameter gradient against the single configurations' added up in extended precision: sums of
    n terms in another order differ by at most n eps of the sum of magnitudes."""
    import torch

    s = W.chain(22)
    sysh = B.grp_create_system(s, B.GRP_FP64 if prec == "fp64" else B.GRP_MIXED)
    q = torch.from_numpy(W.replica_states(s, n_conf, seed=5, spread=0.01)[0]).cuda()
    n = B.grp_param_count(sysh)
    one, tot = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    B.grp_energy_grad(sysh, n_conf, q, None, None, None, tot)
    want, mag = np.zeros(n, np.longdouble), np.zeros(n)
    for b in range(n_conf):
        B.grp_energy_grad(sysh, 1, q[b:b + 1].contiguous(), None, None, None, one)
        v = one.cpu().numpy()
        want += v
        mag += np.abs(v)
    assert np.all(np.abs(tot.cpu().numpy() - want) <= n_conf * 2.0 ** -53 * mag)


@pytest.mark.parametrize("n", [22, 33, 64, 100])
def test_param_gradient_against_autograd(B, n):
    """Mixed-path parameter gradients (positions staged as double-single numbers) far from the origin, where an FP32
    position would have lost the difference: against 64-bit automatic differentiation of the Lennard-Jones and
    torsion terms.  A pair's term is some twenty FP32 operations (1e-6 of its size); the sums have no rounding."""
    import torch

    s = W.chain(n)
    q = W.replica_states(s, 3, seed=8, spread=0.01)[0] + np.array([40.0, -25.0, 60.0])
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    got = torch.empty(B.grp_param_count(sysh), dtype=torch.float64, device="cuda")
    B.grp_energy_grad(sysh, 3, torch.from_numpy(q).cuda(), None, None, None, got)
    sig, eps = (torch.tensor(x, requires_grad=True) for x in (s.sigma, s.epsilon))
    keep = np.ones((n, n), bool)
    keep[s.excl[:, 0], s.excl[:, 1]] = keep[s.excl[:, 1], s.excl[:, 0]] = False
    i, j = (torch.from_numpy(x) for x in np.nonzero(np.triu(keep, 1)))
    x = torch.from_numpy(q)
    s6 = (0.25 * (sig[i] + sig[j]) ** 2 / ((x[:, i] - x[:, j]) ** 2).sum(-1)) ** 3
    e = 4.0 * torch.sqrt(eps[i] * eps[j]) * (s6 * s6 - s6)
    size = [torch.autograd.grad(e.abs().sum(), v, retain_graph=True)[0].abs().numpy().max() for v in (sig, eps)]
    want = [v.numpy() for v in torch.autograd.grad(e.sum(), (sig, eps))]
    for w, g, m in zip(want, (got[:n].cpu().numpy(), got[n:2 * n].cpu().numpy()), size):
        assert np.abs(g - w).max() <= 1e-6 * m


@pytest.mark.parametrize("n", [22, 70, 100])
@pytest.mark.parametrize("shift,grid", [(2.0 ** 6, 2.0 ** -44), (-2.0 ** 9, 2.0 ** -42), (2.0 ** 10, 2.0 ** -41),
                                        (2.0 ** 30, 2.0 ** -20)])
def test_param_gradient_of_shifted_positions(B, n, shift, grid):
    """The mixed path's parameter gradient takes differences of whole FP64 positions: configurations on a grid that
    FP64 still resolves after the shift have the same differences there, and so the same gradient bit for bit (on both
    sides of the range in which the positions are held as FP32 digits)."""
    import torch

    s = W.chain(n)
    sysh = B.grp_create_system(s, B.GRP_MIXED)
    q = np.rint(W.replica_states(s, 16, seed=8, spread=0.01)[0] / grid) * grid
    assert np.array_equal((q + shift) - shift, q)
    here, there = (torch.empty(B.grp_param_count(sysh), dtype=torch.float64, device="cuda") for _ in range(2))
    B.grp_energy_grad(sysh, 16, torch.from_numpy(q).cuda(), None, None, None, here)
    B.grp_energy_grad(sysh, 16, torch.from_numpy(q + shift).cuda(), None, None, None, there)
    assert torch.equal(here, there)
