"""The FP32 strips and the FP64 windows (the automatic choices for periodic members that fill the GPU) against the streaming
kernel: the update of a node is the same sequence of operations, so every result is equal (the
streaming kernel itself is held to the oracle by the parity tests).  Sizes sit at the edges: the
smallest grids, lengths that are not multiples of four, one node more or less than a strip owns
(960 on D1Q5, 672 on D1Q7) and than its lanes hold; step counts below, at and above what one launch
takes (16); one-step calls; a captured call that is replayed."""
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


EQS = {"kdv": (lambda i: W.kdv_burgers(1.0 + 0.2 * i % 5, 0.01 * (i % 9), 0.5 + 0.01 * (i % 50)), 1e-4, 1.15),
       "mkdv": (lambda i: W.mkdv(), 1e-5, 1.2),  # degree 9
       "gkdv": (lambda i: W.gkdv(1.5 + 0.01 * (i % 7)), 1e-4, 1.3),
       "class1": (lambda i: W.class1_real(0.5, 1.0, 1.5, (0.0, 1.0)), 1e-4, 1.3),
       "kawahara": (lambda i: W.kawahara(1.0, 0.5 + 0.01 * (i % 50), -1.0), 1e-4, 2.02)}


def members(eq, sizes):
    make, dt, tau = EQS[eq]
    out = []
    for i, N in enumerate(sizes):
        rng = np.random.default_rng([N, i])
        phi0 = 0.4 + 0.3 * np.cos(2 * np.pi * (np.arange(N) / N + rng.random())) + 0.01 * rng.standard_normal(N)
        out.append(W.Problem(make(i), int(N), 0.1, dt, tau, 0, phi0))
    return out


def sizes(own, K):
    edge = [6, 7, 31, K - 1, K, K + 1, own - 1, own, own + 1, own + K + 3, 2 * own, 2 * own + 5, 4099]
    return edge + list(np.random.default_rng(own).integers(256, 8193, 1000))


def solve(L, ps, kernel, calls):
    return solve_k(L, ps, (kernel, 0), calls)


def solve_k(L, ps, kernel, calls):
    b = L.Batch(ps, precision=L.FP32_DEV).set_kernel(*kernel)
    b.set_phi(np.concatenate([p.phi0 for p in ps]))
    launches = []
    for n in calls:
        n0 = b.kernel_launches()
        b.step(n)
        launches.append(b.kernel_launches() - n0)
    out = b.read_phi()
    b.close()
    return out, launches


@pytest.mark.parametrize("eq,own,K", [("kdv", 960, 32), ("kawahara", 672, 24), ("mkdv", 960, 32), ("gkdv", 960, 32)])
def test_batch(L, eq, own, K):
    ps = members(eq, sizes(own, K))
    a, n = solve(L, ps, L.KERNEL_AUTO, [1, 15, 16, 17, 33])
    b, _ = solve(L, ps, L.KERNEL_STREAM, [82])
    assert n == [1, 1, 1, 2, 3]  # launches of at most 16 steps
    assert np.isfinite(b).all() and np.array_equal(a, b)


@pytest.mark.parametrize("eq,N", [("kdv", (1 << 22) + 3), ("kawahara", (1 << 21) + 1), ("gkdv", (1 << 22) + 1), ("class1", (1 << 22) + 2)])
def test_long_grid(L, eq, N):
    ps = members(eq, [N])
    a, n = solve(L, ps, L.KERNEL_AUTO, [40])
    b, _ = solve(L, ps, L.KERNEL_STREAM, [40])
    assert n == [3] and np.array_equal(a, b)


def test_cubic_flux_on_chip(L):
    """Degree 9 compiled into the on-chip kernel (resident and windows, every CTA class), equal to the
    streaming kernel's run-time degree."""
    ps = members("mkdv", [6, 500, 1000, 1025, 2047, 4000, 4097, 9001])
    a, _ = solve_k(L, ps, (L.KERNEL_ONCHIP, 8), [1, 39])
    b, _ = solve_k(L, ps, (L.KERNEL_STREAM, 0), [40])
    assert np.isfinite(b).all() and np.array_equal(a, b)


@pytest.mark.parametrize("steps", [1, 16, 40])
def test_replayed_capture(L, steps):
    ps = members("kdv", sizes(960, 32))
    want, _ = solve(L, ps, L.KERNEL_STREAM, [3 * steps])
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = L.Batch(ps, precision=L.FP32_DEV)
        b.set_phi(np.concatenate([p.phi0 for p in ps]))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            b.step(steps)
        for _ in range(3):
            g.replay()
        got = b.read_phi()
        b.close()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("eq,sizes64", [("kdv", [200003]), ("kawahara", [150001]), ("kdv", [6, 255, 257, 640, 2048, 2049, 8191] * 16),
                                        ("kawahara", [7, 1000, 1025, 3001] * 24)])
def test_fp64_windows(L, eq, sizes64):
    """FP64 members in windows of a chosen size (equal parts of every member) against the streaming
    kernel, equal; step counts that end in either buffer."""
    ps = members(eq, sizes64)
    phi0 = np.concatenate([p.phi0 for p in ps])
    out = []
    for kernel in (L.KERNEL_AUTO, L.KERNEL_STREAM):
        b = L.Batch(ps, precision=L.FP64).set_kernel(kernel)
        b.set_phi(phi0).step(1).step(16).step(25)
        out.append(b.read_phi())
        b.close()
    assert np.isfinite(out[1]).all() and np.array_equal(out[0], out[1])


@pytest.mark.parametrize("example,count,N,depth", [("4.5", 152, 601, 1), ("4.5", 160, 301, 2), ("4.1", 304, 601, 2), ("4.1", 310, 301, 4),
                                                   ("4.1", 150, 1530, 1)])
def test_fp64_bounded_nodes_a_thread(L, example, count, N, depth):
    """FP64 bounded members on the resident kernel with 3, 4, 5 or 6 nodes a thread, whichever loads
    the schedulers evenly, against 4 nodes a thread and against the streaming step: equal."""
    make, ex, dt, tau, scheme, Wd = {"4.1": (W.ks, W.ks_shock, 1e-3, 1.989, 1 | 0x100, 2),
                                     "4.5": (W.kawahara, W.kawahara_soliton, 1e-4, 2.02, 1, 3)}[example]
    x = W.grid(-0.05 * (N - 1), N, 0.1)
    ps = [W.Problem(make(), N, 0.1, dt, tau + 0.002 * i, 0, ex(x, 0.0), xl=x[0], scheme=scheme, boundary="nee", exact_xt=ex,
                    meta={"depth": depth}) for i in range(count)]
    pb = W.boundary_values(ps[0], Wd, 0, 60)
    out = []
    for args in ((L.KERNEL_AUTO, 0), (L.KERNEL_ONCHIP, 4), (L.KERNEL_STREAM, 0)):
        b = L.Batch(ps, precision=L.FP64).set_kernel(*args)
        b.set_phi(np.tile(ps[0].phi0, count)).step_nee(1, pb[:1]).step_nee(59, np.ascontiguousarray(pb[1:]))
        out.append(b.read_phi())
        b.close()
    assert np.isfinite(out[2]).all() and np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[2])


LINEAR = W.Equation("linear", (1.0, 0.0, 0.1), ((0.0, 1.0), (), (0.0, 1.0)))  # degree 1


@pytest.mark.parametrize("make", [lambda i: (W.mkdv(), 601), lambda i: (W.mkdv() if i % 5 == 0 else W.kdv(), 601),
                                  lambda i: (W.gks_cubic(), 301), lambda i: (W.kdv(), 3001) if i == 7 else (LINEAR, 601)],
                         ids=["cubic", "cubic and quadratic", "degree above 9", "long quadratic, short linear"])
def test_fp64_bounded_other_degrees(L, make):
    """FP64 bounded members whose degree k_bounded has not compiled (all of them, one in five, or the
    short ones beside a longer member of the compiled degree, which streams): as the streaming step."""
    ps = []
    for i in range(304):
        eq, N = make(i)
        phi0 = 0.3 + 0.2 * np.cos(2 * np.pi * (np.arange(N) / N + 0.01 * i))
        ps.append(W.Problem(eq, N, 0.1, 1e-5, 1.1 + 0.001 * i, 0, phi0, boundary="nee", meta={"depth": 2}))
    pb = 0.4 + 0.01 * np.random.default_rng(5).random((40, 4))
    out = []
    for kernel in (L.KERNEL_AUTO, L.KERNEL_STREAM):
        b = L.Batch(ps, precision=L.FP64).set_kernel(kernel)
        b.set_phi(np.concatenate([p.phi0 for p in ps])).step_nee(1, pb[:1]).step_nee(39, np.ascontiguousarray(pb[1:]))
        out.append(b.read_phi())
        b.close()
    assert np.isfinite(out[1]).all() and np.array_equal(out[0], out[1])
