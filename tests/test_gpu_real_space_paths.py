"""Branches of the real-space kernels that the other cells do not reach:
orthogonal lattices whose vectors are not along the axes, shells of 16
primitives (256 primitive pairs an image: the largest positions of a ring entry,
a group number that wraps), and class pairs with d shells at several splits.
Tolerances are 1e-10 times the largest element in FP64 and 1e-7 in the mixed
form, as in the parity tests; between two splits of one plan, whose terms are
the same, a few hundred roundings in FP64 (1e-13) and 1e-9 in the mixed form,
whose FP32 quartets are below 3e-3 (1e-7 of them, some tens of thousands)."""
import numpy as np
import pytest

import synthcells as sc
from oracle import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PAIRS = [(a, b) for a in range(6) for b in range(a, 6)]


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


def oracle_jk(cell):
    D = O.density(cell)
    return (D,) + tuple(O.jk_from_eri(O.eri_tensor(cell), D))


def build(plan, D, sched=None):
    if sched is not None:
        plan.set_schedule(sched)
    Dt = torch.from_numpy(np.ascontiguousarray(D)).cuda()
    J, K = torch.empty_like(Dt), torch.empty_like(Dt)
    plan.build(Dt.data_ptr(), J.data_ptr(), K.data_ptr(), 0)
    torch.cuda.synchronize()
    return J.cpu().numpy(), K.cpu().numpy()


def check(got, ref, precision):
    for g, r in zip(got, ref):
        tol = 1e-10 * max(1.0, np.abs(r).max()) if precision == 0 else 1e-7
        assert np.abs(g - r).max() < tol


def turned(seed, natom, lmax):
    """An orthorhombic cell turned by a rotation about a general axis."""
    cell = sc.small_random_cell(seed, natom=natom, lmax=lmax, skew=False)
    a = np.array([1.0, 2.0, -0.5]) / np.sqrt(5.25)
    X = np.array([[0.0, -a[2], a[1]], [a[2], 0.0, -a[0]], [-a[1], a[0], 0.0]])
    R = np.eye(3) + np.sin(0.7) * X + (1.0 - np.cos(0.7)) * X @ X
    stretch = np.diag([1.0, 1.2, 0.9])
    cell.lattice = cell.lattice @ stretch @ R.T
    cell.positions = cell.positions @ stretch @ R.T
    for s in cell.shells:
        s.center = s.center @ stretch @ R.T
    G = cell.lattice @ cell.lattice.T
    assert np.abs(G - np.diag(np.diag(G))).max() < 1e-12 and np.abs(cell.lattice - np.diag(np.diag(cell.lattice))).max() > 1.0
    cell.name += "turned"
    return cell


@pytest.mark.parametrize("seed,natom,lmax", [(2, 2, 1), (5, 1, 2)])
def test_orthogonal_lattice_off_the_axes(jk, seed, natom, lmax):
    cell = turned(seed, natom, lmax)
    D, Jo, Ko = oracle_jk(cell)
    for precision in (0, 1):
        plan = jk.plan_from_cell(cell, precision=precision)
        for family in (1, 0, 2):
            sched = [(family if (a <= 2 and b <= 2) else 0, 33) for a, b in PAIRS]
            check(build(plan, D, sched), (Jo, Ko), precision)
        plan.close()


@pytest.mark.parametrize("lmax,skew", [(0, False), (1, True)])
@pytest.mark.parametrize("precision", [0, 1])
def test_sixteen_primitives(jk, lmax, skew, precision):
    cell = sc.small_random_cell(7, natom=1, lmax=lmax, skew=skew)
    for s in cell.shells:
        s.exps = np.geomspace(0.25, 12.0, 16)
        s.coefs = np.linspace(0.3, 1.0, 16)
    cell.name += "sixteen"
    D = O.density(cell)
    plan = jk.plan_from_cell(cell, precision=precision)
    assert plan.info()["n_prim_pair_images"] > 200 * plan.info()["n_shell_pairs"]
    ref = build(plan, D, [(0, 16)] * 21)
    for kets in (4, 2048):
        check(build(plan, D, [(1 if (a <= 2 and b <= 2) else 0, kets) for a, b in PAIRS]), ref, precision)
    plan.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_d_class_pairs_at_several_splits(jk, precision):
    """The untuned schedule is compared with the oracle by the parity tests; any
    split gives what it gives, to the rounding of the sums."""
    cell = sc.small_random_cell(3, natom=2, lmax=2)
    D = O.density(cell)
    plan = jk.plan_from_cell(cell, precision=precision)
    ref = build(plan, D)
    for kets in (1, 33, 2048):
        for g, r in zip(build(plan, D, [(1 if (a <= 2 and b <= 2) else 0, kets) for a, b in PAIRS]), ref):
            assert np.abs(g - r).max() < (1e-13 if precision == 0 else 1e-9) * max(1.0, np.abs(r).max()), kets
    plan.close()
