"""jk_energy: odd and even sizes, matrices that are only 8-byte aligned, a
missing J or K, and calls from several threads at once on one plan.  The sums
run over at most 400 products of order one: 1e-11 covers any order of them."""
import threading

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


def matrices(n, shift, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n * n + 1, dtype=torch.float64, device="cuda", generator=g)[shift:shift + n * n] for _ in range(3)]


@pytest.mark.parametrize("natom,lmax", [(1, 0), (1, 2), (2, 1), (2, 2)])
@pytest.mark.parametrize("shift", [0, 1])
def test_energy(jk, natom, lmax, shift):
    cell = sc.small_random_cell(3, natom=natom, lmax=lmax)
    n = cell.nbf
    plan = jk.plan_from_cell(cell)
    D, J, K = matrices(n, shift, n)
    st = torch.cuda.current_stream().cuda_stream
    ej, ek = 0.5 * float((D * J).sum()), -0.25 * float((D * K).sum())
    for j, k in ((J, K), (J, None), (None, K)):
        got = plan.energy(D.data_ptr(), j.data_ptr() if j is not None else 0, k.data_ptr() if k is not None else 0, st)
        assert abs(got[0] - (ej if j is not None else 0.0)) < 1e-11
        assert abs(got[1] - (ek if k is not None else 0.0)) < 1e-11
    plan.close()


def test_energy_from_threads(jk):
    cell = sc.small_random_cell(3, natom=2, lmax=2)
    n = cell.nbf
    plan = jk.plan_from_cell(cell)
    data = [matrices(n, 0, s) for s in range(6)]
    want = [(0.5 * float((D * J).sum()), -0.25 * float((D * K).sum())) for D, J, K in data]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        D, J, K = data[i]
        st = torch.cuda.Stream()
        for _ in range(50):
            got = plan.energy(D.data_ptr(), J.data_ptr(), K.data_ptr(), st.cuda_stream)
            if max(abs(got[0] - want[i][0]), abs(got[1] - want[i][1])) > 1e-11:
                bad.append((i, got, want[i]))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(data))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    plan.close()
    assert not bad, bad[:3]
