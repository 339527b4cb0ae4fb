"""Handles of one equation and precision but of different sizes, stepped from two host threads at
once: they launch the same kernels with different amounts of shared memory."""
import threading

import numpy as np
import pytest

from paper_0907_1720_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0907_1720_gb300 import build as B
    B.build()
    from paper_0907_1720_gb300 import lbhpde
    lbhpde.lib()
    return lbhpde


def periodic(N):
    return W.Problem(W.kdv(), N, 0.1, 1e-5, 1.1, 0, 0.4 + 0.3 * np.cos(2 * np.pi * np.arange(N) / N))


def gkdv(N):
    return W.Problem(W.gkdv(1.5), N, 0.1, 1e-4, 1.3, 0, 0.4 + 0.3 * np.cos(2 * np.pi * np.arange(N) / N))


def bounded(N):
    xl = -0.05 * (N - 1)
    return W.Problem(W.kawahara(), N, 0.1, 1e-4, 2.02, 0, W.kawahara_soliton(W.grid(xl, N, 0.1), 0.0), xl=xl, boundary="nee",
                     exact_xt=W.kawahara_soliton, meta={"depth": 1})


@pytest.mark.parametrize("prec,kernel,make,sizes", [(0, (2, 2), periodic, (64, 2000)), (1, (2, 16), periodic, (64, 8000)),
                                                    (1, (0, 0), gkdv, (64, 2500)), (0, (2, 4), bounded, (24, 1000))],
                         ids=["on-chip", "16-node", "automatic", "bounded"])
def test_two_threads(L, prec, kernel, make, sizes):
    calls, errors, got = 2000, [], {}
    want = {}
    for N in sizes:
        p = make(N)
        pb = W.boundary_values(p, 3, 0, 1) if p.boundary == "nee" else None
        with torch.cuda.stream(torch.cuda.Stream()):
            s = L.Solver.for_problem(p, precision=prec).set_kernel(*kernel).set_phi(p.phi0)
            for _ in range(calls):
                s.step(1) if pb is None else s.step_nee(1, pb)
            want[N] = s.read_phi()
            s.close()
    start = threading.Barrier(2)

    def work(N):
        try:
            p = make(N)
            with torch.cuda.stream(torch.cuda.Stream()):
                pb = torch.from_numpy(W.boundary_values(p, 3, 0, 1)).cuda() if p.boundary == "nee" else None
                s = L.Solver.for_problem(p, precision=prec).set_kernel(*kernel).set_phi(p.phi0)
                start.wait(timeout=60)
                for _ in range(calls):
                    s.step(1) if pb is None else s.step_nee(1, pb)
                got[N] = s.read_phi()
                s.close()
        except Exception as e:  # reported below: an assertion in a thread would be lost
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(N,)) for N in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for N in sizes:
        assert np.isfinite(want[N]).all() and np.array_equal(got[N], want[N])
