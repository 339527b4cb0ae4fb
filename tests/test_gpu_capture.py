"""Captured calls, replayed: a call has to end in the buffer it began in, whatever kernels a batch's
members take and however many launches the call is.  Each against the streaming kernel's steps
launched one by one, equal bit for bit."""
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


def periodic(N, i=0):
    phi0 = 0.4 + 0.3 * np.cos(2 * np.pi * (np.arange(N) / N + 0.1 * i))
    return W.Problem(W.kdv(), int(N), 0.1, 1e-5, 1.1, 0, phi0)


def bounded(N):
    xl = -0.05 * (N - 1)
    return W.Problem(W.ks(), N, 0.1, 1e-3, 1.989, 0, W.ks_shock(W.grid(xl, N, 0.1), 0.0), xl=xl, scheme=1 | 0x100, boundary="nee",
                     exact_xt=W.ks_shock, meta={"depth": 2})


BATCHES = {  # (precision, members): windows or strips, residents, each beside bounded ones
    "fp32 strips, one bounded warp": (1, lambda: [periodic(N, i) for i, N in enumerate([4000, 700, 9001] * 150)] + [bounded(601)] * 3),
    "fp32 windows and residents": (1, lambda: [periodic(20000), periodic(300, 1)] + [bounded(601)]),
    "fp64 windows": (0, lambda: [periodic(N, i) for i, N in enumerate([200003, 300])] + [bounded(601)] * 3),
    "fp64 windows, streamed bounded": (0, lambda: [periodic(100003), bounded(3001), bounded(301)]),
}


def replayed(L, ps, prec, kernel, steps, phib, replays=3):
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = L.Batch(ps, precision=prec).set_kernel(*kernel)
        b.set_phi(np.concatenate([p.phi0 for p in ps]))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            b.step(steps) if phib is None else b.step_nee(steps, phib)
        for _ in range(replays):
            g.replay()
        got = b.read_phi()
        b.close()
    return got


def streamed(L, ps, prec, steps, phib, calls=3):
    b = L.Batch(ps, precision=prec).set_kernel(L.KERNEL_STREAM)
    b.set_phi(np.concatenate([p.phi0 for p in ps]))
    for _ in range(calls):
        b.step(steps) if phib is None else b.step_nee(steps, phib)
    out = b.read_phi()
    b.close()
    return out


@pytest.mark.parametrize("steps", [1, 2, 3, 17])
@pytest.mark.parametrize("name", list(BATCHES))
def test_mixed_batches(L, name, steps):
    prec, make = BATCHES[name]
    ps = make()
    phib = torch.from_numpy(W.boundary_values(bounded(601), 2, 0, steps)).cuda()
    got = replayed(L, ps, prec, (L.KERNEL_AUTO,), steps, phib)
    want = streamed(L, ps, prec, steps, phib)
    assert np.isfinite(want).all() and np.array_equal(got, want)


@pytest.mark.parametrize("steps", [1, 2, 3, 7])
@pytest.mark.parametrize("prec,K", [(0, 4), (1, 8)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("per_launch", [1, 2])
def test_windows_of_few_steps_a_launch(L, per_launch, prec, K, steps):
    """Windows of one or two steps a launch (asked for), with residents beside them."""
    ps = [periodic(20011), periodic(300, 1), periodic(5000, 2)]
    got = replayed(L, ps, prec, (L.KERNEL_ONCHIP, K, per_launch), steps, None)
    want = streamed(L, ps, prec, steps, None)
    assert np.isfinite(want).all() and np.array_equal(got, want)


def test_tuned_one_step_a_launch(L):
    """The same from a tuned pair of one step a launch (a degree that nothing else here uses)."""
    eq = W.Equation("linear", (1.0, 0.0, 0.1), ((0.0, 1.0), (), (0.0, 1.0)))
    ps = [W.Problem(eq, 9001 + 11 * i, 0.1, 1e-5, 1.1, 0, periodic(9001 + 11 * i).phi0) for i in range(2)]
    want = streamed(L, ps, 0, 3, None)
    L.set_tuning(L.FP64, 5, 1, 4, 1)
    try:
        got = replayed(L, ps, 0, (L.KERNEL_HALO,), 3, None)
    finally:
        L.set_tuning(L.FP64, 5, 1, 4, 64)  # the untuned pair, for the tests that follow
    assert np.isfinite(want).all() and np.array_equal(got, want)


@pytest.mark.parametrize("steps", [1, 7, 8, 40])
def test_unequal_bounded_members(L, steps):
    """Bounded members whose launches run side by side, captured and not."""
    ps = [bounded(N) for N in (97, 150, 231, 301, 420, 601, 700, 850, 1000, 601)] * 20  # one warp each, every number of nodes a lane
    phib = torch.from_numpy(W.boundary_values(bounded(601), 2, 0, steps)).cuda()
    want = streamed(L, ps, 1, steps, phib)
    got = replayed(L, ps, 1, (L.KERNEL_AUTO,), steps, phib)
    b = L.Batch(ps, precision=1)
    b.set_phi(np.concatenate([p.phi0 for p in ps]))
    for _ in range(3):
        b.step_nee(steps, phib)
    assert np.isfinite(want).all() and np.array_equal(got, want) and np.array_equal(b.read_phi(), want)
    b.close()


def kawahara(N):
    return W.Problem(W.kawahara(), int(N), 0.1, 1e-4, 2.02, 0, 0.4 + 0.3 * np.cos(2 * np.pi * np.arange(N) / N))


LATTICES = {  # two groups with windows or strips of depths of their own, residents beside them
    "fp64 windows": (0, (0, 0, 0), lambda: [periodic(200003), periodic(300, 1), kawahara(100003), kawahara(500)]),
    "fp32 strips": (1, (0, 0, 0), lambda: [periodic(700001), kawahara(600001)]),
    "fp32 strips and windows": (1, (0, 0, 0), lambda: [periodic(700001), kawahara(20011), kawahara(300)]),
    "one step a launch": (0, (3, 4, 1), lambda: [periodic(9001), kawahara(5003)]),
}


@pytest.mark.parametrize("steps", [1, 2, 3, 17, 40])
@pytest.mark.parametrize("name", list(LATTICES))
def test_two_lattices(L, name, steps):
    """The windows of the two lattices run side by side and end in one buffer, captured or not."""
    prec, kernel, make = LATTICES[name]
    ps = make()
    want = streamed(L, ps, prec, steps, None)
    assert np.isfinite(want).all() and np.array_equal(replayed(L, ps, prec, kernel, steps, None), want)
    b = L.Batch(ps, precision=prec).set_kernel(*kernel)
    b.set_phi(np.concatenate([p.phi0 for p in ps]))
    for _ in range(3):
        b.step(steps)
    assert np.array_equal(b.read_phi(), want)
    b.close()
