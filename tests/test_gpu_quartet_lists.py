"""Lists of large quartets of small mixed plans, which run several class pairs at
once: the plan's workspace (what a server admits it by) is no larger than with
one list, and every list holds its class pairs.

The limits are the bytes of these plans with one list of 8-byte entries.  With a
switch of 1e-300 every quartet whose estimate does not underflow goes to the
lists; what is left of the mixed path is the split exchange and the double-float
structure factors, some 1e-11, hence 1e-9 against the FP64 build."""
import numpy as np
import pytest

import synthcells as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELLS = {
    "tiny": (sc.tiny_cell, 311018788),
    "skewed_spd": (lambda: sc.small_random_cell(1, natom=2, lmax=2, skew=True), 382144468),
    "water5": (lambda: sc.water_cell(5, (29.94 * 5) ** (1.0 / 3.0), n_occ=20), 627094200),
    "diamond1": (lambda: sc.diamond_cell(1), 499547580),
    "diamond1_soft": (lambda: sc.diamond_cell(1, omega=0.4), 288255684),  # the G chunk gives up four vectors
}


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


@pytest.mark.parametrize("name", list(CELLS))
def test_workspace(jk, name):
    make, limit = CELLS[name]
    plan = jk.plan_from_cell(make(), precision=jk.JK_MIXED)
    got = plan.info()["workspace_bytes"]
    plan.close()
    assert got <= limit, (got, limit)


@pytest.mark.parametrize("name", ["tiny", "skewed_spd"])
@pytest.mark.parametrize("want_k", [True, False])
def test_every_quartet_listed(jk, name, want_k):
    cell = CELLS[name][0]()
    D, out = None, []
    for precision in (jk.JK_FP64, jk.JK_MIXED):
        plan = jk.plan_from_cell(cell, precision=precision, mixed_switch=1e-300)
        if D is None:
            S = torch.empty((cell.nbf, cell.nbf), dtype=torch.float64, device="cuda")
            plan.overlap(S.data_ptr(), 0)
            torch.cuda.synchronize()
            D = torch.from_numpy(sc.density_from_overlap(cell.orbital_guess(), S.cpu().numpy())).cuda()
        J, K = torch.empty_like(D), torch.zeros_like(D)
        for _ in range(2):
            plan.build(D.data_ptr(), J.data_ptr(), K.data_ptr() if want_k else 0, 0)
        torch.cuda.synchronize()
        c = plan.counters()
        out.append((J.cpu().numpy(), K.cpu().numpy(), c))
        plan.close()
    assert out[1][2]["list_overflow"] == 0
    assert out[1][2]["quartets_fp64"] > 0.5 * (out[1][2]["quartets_fp64"] + out[1][2]["quartets_fp32"])
    for ref, got in zip(out[0][:2], out[1][:2]):
        assert np.abs(got - ref).max() < 1e-9
