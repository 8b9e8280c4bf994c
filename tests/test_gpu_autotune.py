"""jk_autotune keeps the untuned schedule unless a candidate is faster over the
class: the tuned tiles of the 64-water box are not slower than the untuned ones
(run-to-run differences are below 1 %; 5 % allowed), the choices come back from
the cache file, and a damaged line leaves the untuned schedule."""
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


def density(jk, plan, cell):
    S = torch.empty((cell.nbf, cell.nbf), dtype=torch.float64, device="cuda")
    plan.overlap(S.data_ptr(), 0)
    torch.cuda.synchronize()
    return torch.from_numpy(sc.density_from_overlap(cell.orbital_guess(), S.cpu().numpy())).cuda()


def tiles(plan, D):
    J, K = torch.empty_like(D), torch.empty_like(D)
    best = 1e30
    for _ in range(3):
        plan.build(D.data_ptr(), J.data_ptr(), K.data_ptr(), 0)
        best = min(best, plan.build_times()["real_tiles"][0])
    return best


def test_tuned_is_not_slower(jk, tmp_path):
    cell = sc.config(2)
    plan = jk.plan_from_cell(cell, precision=jk.JK_MIXED)
    D = density(jk, plan, cell)
    untuned = tiles(plan, D)
    path = str(tmp_path / "cache.txt")
    chosen = plan.autotune(D.data_ptr(), cache_path=path)
    tuned = tiles(plan, D)
    again = plan.autotune(D.data_ptr(), cache_path=path)
    plan.close()
    print("tiles: untuned %.1f ms, tuned %.1f ms" % (untuned, tuned), chosen)
    assert tuned <= 1.05 * untuned, (untuned, tuned, chosen)
    assert again == chosen


def test_damaged_cache_line(jk, tmp_path):
    cell = sc.tiny_cell()
    plan = jk.plan_from_cell(cell)
    D = density(jk, plan, cell)
    path = tmp_path / "cache.txt"
    plan.autotune(D.data_ptr(), cache_path=str(path))
    lines = path.read_text().split("\n")
    path.write_text("\n".join(l.rsplit(" ", 1)[0] + " 0" if l else l for l in lines))
    own = plan.autotune(D.data_ptr(), cache_path=str(path))  # 0: the untuned schedule
    path.write_text("\n".join(l.rsplit(" ", 1)[0] + " %d" % (7 * 65536 + 3) if l else l for l in lines))
    assert plan.autotune(D.data_ptr(), cache_path=str(path)) == own
    assert all(f in (0, 1, 2) and k >= 1 for f, k in own)
    plan.close()
