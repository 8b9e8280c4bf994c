"""jk_one_electron gives the same bits when it is repeated: cells with many
images a shell pair, with charges in 8 and in 32 lanes, and the form of the
reciprocal part for reciprocal vectors with an integer coordinate above 64."""
import numpy as np
import pytest

import synthcells as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


def elongated():
    cell = sc.small_random_cell(2, 1, 1, False)
    lat = np.array(cell.lattice, dtype=float)
    lat[2] *= 90.0 / np.linalg.norm(lat[2])
    cell.lattice = lat
    return cell


CELLS = {"tiny": sc.tiny_cell, "skewed_spd": lambda: sc.small_random_cell(1, natom=2, lmax=2, skew=True), "elongated": elongated,
         "water8": lambda: sc.water_cell(8, (29.94 * 8) ** (1.0 / 3.0), n_occ=32)}


@pytest.mark.parametrize("name", list(CELLS))
def test_repeated_calls_agree_to_the_bit(jk, name):
    cell = CELLS[name]()
    plan = jk.plan_from_cell(cell)
    Z, xyz = sc.nuclear_charges(cell), cell.positions
    out = []
    for _ in range(12):
        T = torch.empty((cell.nbf, cell.nbf), dtype=torch.float64, device="cuda")
        V = torch.empty_like(T)
        plan.one_electron(Z, xyz, T.data_ptr(), V.data_ptr(), 0)
        out.append((T, V))
    alone = torch.empty_like(T)
    plan.one_electron(Z, xyz, alone.data_ptr(), 0, 0)
    plan.close()
    assert all(torch.equal(T, out[0][0]) and torch.equal(V, out[0][1]) for T, V in out)
    assert torch.equal(alone, out[0][0])
    assert torch.isfinite(out[0][0]).all() and torch.isfinite(out[0][1]).all()
