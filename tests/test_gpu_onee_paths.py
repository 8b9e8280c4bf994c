"""The branches of jk_one_electron: few and many charges (8 or 32 lanes per
primitive pair) and the two forms of the reciprocal part (phase tables, or the
structure-factor slab when a reciprocal vector has an integer coordinate above
64).  Tolerance 1e-10, the FP64 parity bound of test_gpu_one_electron.py."""
import numpy as np
import pytest

import synthcells as sc
from oracle import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


def attraction(plan, n, Z, xyz):
    T = torch.empty((n, n), dtype=torch.float64, device="cuda")
    V = torch.full_like(T, float("nan"))
    plan.one_electron(np.ascontiguousarray(Z), np.ascontiguousarray(xyz), T.data_ptr(), V.data_ptr(), 0)
    return V.cpu().numpy()


@pytest.mark.parametrize("seed,natom,lmax,skew", [(2, 2, 2, True), (1, 1, 1, False)])
@pytest.mark.parametrize("count", [16, 17, 33])
def test_attraction_is_linear_in_the_charges(jk, seed, natom, lmax, skew, count):
    cell = sc.small_random_cell(seed, natom, lmax, skew)
    rng = np.random.default_rng(count)
    Z = rng.uniform(-3.0, 3.0, count)
    xyz = rng.uniform(0.0, 1.0, (count, 3)) @ np.asarray(cell.lattice)
    plan = jk.plan_from_cell(cell)
    whole = attraction(plan, cell.nbf, Z, xyz)
    parts = sum(attraction(plan, cell.nbf, Z[i:i + 5], xyz[i:i + 5]) for i in range(0, count, 5))
    plan.close()
    assert np.array_equal(whole, whole.T)
    assert np.abs(whole - parts).max() < TOL


@pytest.mark.parametrize("edge", [20.0, 90.0])  # largest integer coordinate of a reciprocal vector below and above 64
def test_elongated_cell_matches_oracle(jk, edge):
    cell = sc.small_random_cell(2, 1, 1, False)
    lat = np.array(cell.lattice, dtype=float)
    lat[2] *= edge / np.linalg.norm(lat[2])
    cell.lattice = lat
    plan = jk.plan_from_cell(cell)
    V = attraction(plan, cell.nbf, sc.nuclear_charges(cell), cell.positions)
    plan.close()
    assert np.abs(V - O.nuclear(cell)).max() < TOL
