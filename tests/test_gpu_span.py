"""The one-warp kernel of bounded FP32 members (k_span, the automatic choice for D1Q5 of 96 to 1024
nodes at depth 2 and D1Q7 of 129 to 768 at depths 1 and 2, unless the batch is small) against k_bounded's four-nodes-a-thread variant, with which it
shares no code of the ends: the same sequence of operations a node, so every result is equal bit for
bit.  One batch for each number of nodes a lane holds, with members of every remainder (the
right end's registers), step counts below, at and above the eight steps whose boundary values are
staged at once, in one call and in several."""
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


EQS = {"ks": (W.ks, W.ks_shock, 1e-3, 1.989, 1 | 0x100, 2),                   # D1Q5
       "kawahara": (W.kawahara, W.kawahara_soliton, 1e-4, 2.02, 1, 3)}  # D1Q7


def problem(N, depth=2, eq="ks"):
    make, ex, dt, tau, scheme, _ = EQS[eq]
    xl = -0.05 * (N - 1)
    return W.Problem(make(), N, 0.1, dt, tau, 0, ex(W.grid(xl, N, 0.1), 0.0), xl=xl, scheme=scheme, boundary="nee",
                     exact_xt=ex, meta={"depth": depth})


def solve(L, probs, kernel, K, calls, eq="ks"):
    """phi after the step counts in `calls`, and the launches of the last call."""
    steps, Wd = sum(calls), EQS[eq][5]
    one = {}
    for p in probs:
        if p.N not in one:
            one[p.N] = W.boundary_values(p, Wd, 0, steps).reshape(steps, 2 * Wd)
    b = L.Batch(probs, precision=L.FP32_DEV).set_kernel(kernel, K)
    b.set_phi(np.concatenate([p.phi0 for p in probs]))
    done = 0
    for n in calls:
        n0 = b.kernel_launches()
        b.step_nee(n, np.concatenate([one[p.N][done:done + n].ravel() for p in probs]), 2 * Wd * n)
        done += n
    launches = b.kernel_launches() - n0
    got = b.read_phi()
    b.close()
    return got, launches


@pytest.mark.parametrize("calls", [(7,), (8, 1), (1, 19)], ids=str)
@pytest.mark.parametrize("K", [4, 8, 12, 16, 20, 24, 28, 32])
def test_span_matches_bounded_bitwise(L, K, calls):
    sizes = [n for n in range(32 * (K - 4) + 1, 32 * K + 1) if n >= max(96, 0.6 * 32 * K)]
    sizes = sizes[:40] + sizes[-33:]  # every remainder, at both ends of the range
    probs = [problem(n) for n in sizes] * (40 if K <= 12 else 16)
    got, launches = solve(L, probs, L.KERNEL_AUTO, 0, calls)
    want, _ = solve(L, probs, L.KERNEL_ONCHIP, 4, calls)
    assert launches == 1
    assert np.isfinite(got).all() and np.array_equal(got, want)


@pytest.mark.parametrize("calls", [(4,), (5, 1), (1, 13)], ids=str)
@pytest.mark.parametrize("K", [8, 12, 16, 20, 24])
def test_span_d1q7_matches_bounded_bitwise(L, K, calls):
    """D1Q7: three outer nodes an end, depths 1 and 2, five steps' boundary values at once."""
    sizes = [n for n in range(32 * (K - 4) + 1, 32 * K + 1) if n >= max(129, 0.6 * 32 * K)]
    sizes = sizes[:40] + sizes[-33:]
    probs = [problem(n, 1 + (n + r) % 2, "kawahara") for r in range(40 if K <= 12 else 18) for n in sizes]
    got, launches = solve(L, probs, L.KERNEL_AUTO, 0, calls, "kawahara")
    want, _ = solve(L, probs, L.KERNEL_ONCHIP, 4, calls, "kawahara")
    assert launches == 1
    assert np.isfinite(got).all() and np.array_equal(got, want)


def test_span_beside_other_kernels(L):
    """Members of other depths and sizes keep their kernels (k_ring_nee) in the same batch."""
    sizes = [(601, 2), (601, 3), (95, 2), (96, 2), (129, 2), (1024, 2), (1025, 2), (300, 1)]
    probs = [problem(n, d) for n, d in sizes] * 100
    got, _ = solve(L, probs, L.KERNEL_AUTO, 0, (11, 6))
    want, _ = solve(L, probs, L.KERNEL_ONCHIP, 4, (11, 6))
    o = 0
    for p, (n, d) in zip(probs, sizes * 100):
        a, b = got[o:o + n], want[o:o + n]
        # k_ring_nee adds a node's differences in another order: an ulp of phi a step at most
        ok = np.array_equal(a, b) if d == 2 and n in (96, 601, 1024) else np.abs(a - b).max() <= 17 * 5 * 2.0 ** -23 * np.abs(b).max()
        assert ok, (n, d)
        o += n
