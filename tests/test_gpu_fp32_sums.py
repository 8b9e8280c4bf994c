"""FP32 sums of heavily contracted quartets: with 16 primitives a shell, a block
adds 65536 terms.  Every quartet in FP32 (mixed_switch 1e30) against the FP64
build, one atom with s, s and p, or s, p and d shells; the bound is the parity
bound of test_gpu_mixed_parity.py for forced FP32, 16 units of the last place of
the largest element, whatever the contraction: the rounding of the sums must not
grow with their length."""
import numpy as np
import pytest

import synthcells as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_FP32_REL = 16 * 2.0 ** -24


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


@pytest.mark.parametrize("lmax,nprim", [(0, 16), (1, 16), (1, 6), (2, 4)])
def test_long_contractions(jk, lmax, nprim):
    cell = sc.small_random_cell(7, natom=1, lmax=lmax, skew=False)
    for s in cell.shells:
        s.exps = np.geomspace(0.25, 12.0, nprim)
        s.coefs = np.linspace(0.3, 1.0, nprim)
    out = []
    D = None
    for precision in (jk.JK_FP64, jk.JK_MIXED):
        plan = jk.plan_from_cell(cell, precision=precision, mixed_switch=1e30)
        if D is None:
            S = torch.empty((cell.nbf, cell.nbf), dtype=torch.float64, device="cuda")
            plan.overlap(S.data_ptr(), 0)
            torch.cuda.synchronize()
            D = torch.from_numpy(sc.density_from_overlap(cell.orbital_guess(), S.cpu().numpy())).cuda()
        J, K = torch.empty_like(D), torch.empty_like(D)
        plan.build(D.data_ptr(), J.data_ptr(), K.data_ptr(), 0)
        torch.cuda.synchronize()
        out.append((J.cpu().numpy(), K.cpu().numpy()))
        plan.close()
    for name, ref, got in zip("JK", *out):
        scale = max(1.0, np.abs(ref).max())
        print("lmax %d nprim %d %s: %.2f ulp" % (lmax, nprim, name, np.abs(got - ref).max() / scale * 2.0 ** 24))
        assert np.abs(got - ref).max() < TOL_FP32_REL * scale, name
