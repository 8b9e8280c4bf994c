"""Real-space tile kernels at the edges of their work split: any number of
kets per warp, bras with more primitive pairs than one screening round holds
(17 to 36), cells with fewer image quartets than warps.

The reference is the lane-per-bra family (no split of a bra's kets over warps,
no batches) on the same plan, whose terms are the same up to those on the edge
of a screening sphere (each below a tenth of the 1e-12 threshold) and the
order of the sums: 1e-10 times the largest element in FP64, the parity bound
1e-7 in the mixed form.  Class pairs with a d shell have one kernel; for them
the split alone varies.
"""
import numpy as np
import pytest

import synthcells as sc
from oracle import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


def wide_cell(natom, lmax, skew, nprim):
    """A small cell whose shells have nprim primitives (nprim^2 per image)."""
    c = sc.small_random_cell(7, natom=natom, lmax=lmax, skew=skew)
    for s in c.shells:
        s.exps = np.geomspace(0.25, 12.0, nprim)
        s.coefs = np.linspace(0.3, 1.0, nprim)
    c.name = "wide%d%d%d%d" % (natom, lmax, skew, nprim)
    return c


@pytest.mark.parametrize("natom,lmax,skew,nprim", [(1, 1, True, 5), (2, 0, False, 6), (1, 2, False, 2)])
@pytest.mark.parametrize("precision", [0, 1])
def test_any_split_gives_the_same(jk, natom, lmax, skew, nprim, precision):
    cell = wide_cell(natom, lmax, skew, nprim)
    Dt = torch.from_numpy(O.density(cell)).cuda()
    plan = jk.plan_from_cell(cell, precision=precision)

    def build(family, kets):
        plan.set_schedule([(family if (a <= 2 and b <= 2) else 0, kets) for a in range(6) for b in range(a, 6)])
        J, K = torch.empty_like(Dt), torch.empty_like(Dt)
        plan.build(Dt.data_ptr(), J.data_ptr(), K.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return J.cpu().numpy(), K.cpu().numpy()

    refs = build(0, 16)
    for kets in (1, 7, 33, 2048):
        for got, ref in zip(build(1, kets), refs):
            tol = 1e-10 * max(1.0, np.abs(ref).max()) if precision == 0 else 1e-7
            assert np.abs(got - ref).max() < tol, kets
    plan.close()
