"""jk_build_times of plans whose phases run on several streams: no phase is
longer than the build, and the tile kernels and list passes lie inside real
space.  Event times carry microseconds: 2 % and 0.02 ms."""
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


def small():
    return sc.water_cell(5, (29.94 * 5) ** (1.0 / 3.0), n_occ=20)


@pytest.mark.parametrize("make,precision", [(small, 1), (small, 0), (lambda: sc.diamond_cell(1), 1)])
def test_phases_of_a_small_plan(jk, make, precision):
    cell = make()
    plan = jk.plan_from_cell(cell, precision=precision)
    D = 0.1 * torch.eye(cell.nbf, dtype=torch.float64, device="cuda") + 0.01
    J, K = torch.empty_like(D), torch.empty_like(D)
    for _ in range(3):
        plan.build(D.data_ptr(), J.data_ptr(), K.data_ptr(), 0)
    t = {p: v[0] for p, v in plan.build_times().items() if p != "mma_flops"}
    plan.close()

    def within(a, b):
        return t[a] <= 1.02 * t[b] + 0.02

    assert all(within(p, "total") for p in t), t
    assert within("real_tiles", "real_space") and within("real_fp64_list", "real_space"), t
    assert t["real_tiles"] > 0 and t["recip_k"] > 0, t
