"""jk_energy where its launch has many blocks, from several threads at once on
one plan, and in a thread that still carries the error of an earlier CUDA call
(an allocation that was refused, which faults nothing): the call is judged by
its own launch and always waits for it.  The sums run over 43 thousand
products of order one: 1e-9 covers any order of them."""
import ctypes
import threading

import numpy as np
import pytest

import synthcells as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-9


@pytest.fixture(scope="module")
def jk():
    from paper_2410_22278_gb300 import build, jk

    build.build()
    assert torch.cuda.is_available()
    return jk


@pytest.fixture(scope="module")
def plan(jk):
    p = jk.plan_from_cell(sc.water_cell(16, (29.94 * 16) ** (1.0 / 3.0), n_occ=64))
    assert p.nbf >= 200  # 43 blocks
    yield p
    p.close()


def matrices(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n * n, dtype=torch.float64, device="cuda", generator=g) for _ in range(3)]


def expected(D, J, K):
    return 0.5 * float((D * J).sum()), -0.25 * float((D * K).sum())


def leave_error():
    """A refused allocation; the runtime keeps its error for this thread."""
    rt = ctypes.CDLL("libcudart.so.13")  # the one that is loaded already
    rt.cudaMalloc.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), 1 << 60) != 0
    assert rt.cudaPeekAtLastError() != 0


def clear_error():
    ctypes.CDLL("libcudart.so.13").cudaGetLastError()


def test_error_of_an_earlier_call(jk, plan):
    D, J, K = matrices(plan.nbf, 1)
    want = expected(D, J, K)
    st = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    leave_error()
    try:
        got = plan.energy(D.data_ptr(), J.data_ptr(), K.data_ptr(), st)
    finally:
        clear_error()
    assert max(abs(got[0] - want[0]), abs(got[1] - want[1])) < TOL


def test_error_of_an_earlier_call_without_allocation(jk, plan):
    D, J, K = matrices(plan.nbf, 2)
    want = expected(D, J, K)
    st = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    leave_error()
    try:
        got = plan.energy_noalloc(D.data_ptr(), J.data_ptr(), K.data_ptr(), st)
    finally:
        clear_error()
    assert max(abs(got[0] - want[0]), abs(got[1] - want[1])) < TOL


def test_threads_with_and_without_one(jk, plan):
    data = [matrices(plan.nbf, 10 + s) for s in range(6)]
    want = [expected(*d) for d in data]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        D, J, K = data[i]
        st = torch.cuda.Stream()
        try:
            for _ in range(100):
                if i % 2:
                    leave_error()
                got = plan.energy(D.data_ptr(), J.data_ptr(), K.data_ptr(), st.cuda_stream)
                if max(abs(got[0] - want[i][0]), abs(got[1] - want[i][1])) > TOL:
                    bad.append((i, got, want[i]))
        except Exception as e:
            bad.append((i, e))
        finally:
            clear_error()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(data))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:3]


def test_refused_allocation_of_the_library(jk, plan):
    """The error of a failed allocation is reported by its call and not kept."""
    cell = sc.water_cell(16, (29.94 * 16) ** (1.0 / 3.0), n_occ=64)
    big = jk.plan_from_cell(cell, omega=3.0)
    need = 16 * cell.nbf ** 2 * big.info()["n_g"]  # the reciprocal cache
    assert need > 1.2 * torch.cuda.get_device_properties(0).total_memory
    with pytest.raises(jk.JkError) as e:
        big.cache(2 * need)
    assert e.value.status == jk.JK_ERR_OOM
    assert ctypes.CDLL("libcudart.so.13").cudaPeekAtLastError() == 0
    D, J, K = matrices(plan.nbf, 3)
    got = plan.energy(D.data_ptr(), J.data_ptr(), K.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert np.allclose(got, expected(D, J, K), rtol=0, atol=TOL)
    big.close()
