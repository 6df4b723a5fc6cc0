"""The streamed block passes of the Arnoldi step (dots in fixed point on the
integer pipe) against the MGS loop in numpy.

Vector lengths around the passes' tile (256 elements) and grid edges, every
last-block size, values that force new fixed-point scales (magnitudes growing
along the vector, isolated large entries, zeros), operands that no bulk copy
can start on (8-byte aligned: the register kernels), infinities and NaN, and
the 8-vector blocks of GMRES over a long cycle.

Tolerance of the coefficients: MGS in FP64 gives each h_i to within a few
rounding errors of |w| |v_i| = |w|; both sides accumulate at most N of them in
trees or chains of length < 1000, so 1e-12 |w| holds with margin, and w and
v_{j+1} likewise to 1e-11 (division by the norm of what is left of w)."""
import numpy as np
import pytest
import torch

import rt_workloads as W
from gpu_util import problem, to_dev, to_host

pytestmark = pytest.mark.gpu


def _mgs(Q, w):
    h = []
    for v in Q:
        h.append(np.dot(w, v))
        w = w - h[-1] * v
    h.append(np.linalg.norm(w))
    return np.array(h), w


def _values(kind, N, rng):
    w = rng.standard_normal(N)
    if kind == "growing":
        w *= np.exp(np.linspace(-30.0, 10.0, N))
    elif kind == "spikes":
        w[rng.integers(0, N, 5)] *= 1e9
    elif kind == "zeros":
        w[: N // 2] = 0.0
        w[N // 2:: 3] = 0.0
    elif kind == "tiny":
        w *= 1e-290
    return w


def _step(P, N, j, kind, offset=0, seed=0):
    rng = np.random.default_rng(seed)
    Q = []
    for i in range(j + 1):
        v = _values("growing" if kind == "growing" and i % 2 else "normal", N, rng)
        for _ in range(2):
            for u in Q:
                v = v - np.dot(u, v) * u
        Q.append(v / np.linalg.norm(v))
    w0 = _values(kind, N, rng)
    gram = np.zeros((j + 2, 4))
    for i in range(1, j + 1):
        for d in range(1, min(i, 3) + 1):
            gram[i, d] = Q[i] @ Q[i - d]
    buf = torch.zeros((j + 2) * N + 2, dtype=torch.float64, device="cuda")
    Vd = buf[offset: offset + (j + 2) * N]
    Vd[: (j + 1) * N] = to_dev(np.concatenate(Q))
    wbuf = torch.zeros(N + 2, dtype=torch.float64, device="cuda")
    wd = wbuf[offset: offset + N]
    wd.copy_(to_dev(w0))
    h = to_host(P.arnoldi_bmgs(Vd, j, wd, to_dev(gram.reshape(-1))))
    P.check()
    href, w = _mgs(Q, w0)
    s = np.abs(w0).max() * np.linalg.norm(w0 / np.abs(w0).max())   # |w0| without underflow of its square
    np.testing.assert_allclose(h, href, rtol=0, atol=1e-12 * s)
    np.testing.assert_allclose(to_host(wd), w, rtol=0, atol=1e-11 * s)
    if href[-1] > 0.0:   # (the square of the norm underflows for the tiny values, on both sides)
        np.testing.assert_allclose(to_host(Vd)[(j + 1) * N:], w / href[-1], rtol=0, atol=1e-11 * s / href[-1])


# N = 2 Ns Nmu Nnu: below, at and just past one tile; several tiles; more tiles than CTAs
@pytest.mark.parametrize("Ns,Nmu,Nnu", [(2, 2, 2), (21, 2, 3), (32, 2, 2), (43, 2, 3), (64, 4, 2), (43, 2, 6),
                                        (37, 6, 33), (100, 16, 61)])
@pytest.mark.parametrize("j", [0, 3, 4, 6, 13])
def test_pass_sizes(Ns, Nmu, Nnu, j):
    P = problem(W.slab(Ns, Nmu, Nnu, 1e-4, 1e6, 6.0))
    if j + 2 > P.N:
        j = P.N - 3
    _step(P, P.N, j, "normal", seed=j)


@pytest.mark.parametrize("kind", ["growing", "spikes", "zeros", "tiny"])
@pytest.mark.parametrize("offset", [0, 1])   # 1: 8-byte aligned operands
def test_pass_values(kind, offset):
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    _step(P, P.N, 9, kind, offset, seed=3)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_pass_not_finite(bad):
    """A non-finite w gives non-finite coefficients, as the FP64 products do."""
    P = problem(W.slab(37, 6, 33, 1e-4, 1e6, 6.0))
    N, j = P.N, 5
    rng = np.random.default_rng(0)
    V = torch.zeros((j + 2) * N, dtype=torch.float64, device="cuda")
    V[: (j + 1) * N] = to_dev(rng.standard_normal((j + 1) * N) / np.sqrt(N))
    w0 = rng.standard_normal(N)
    w0[N // 3] = bad
    v0 = to_host(V)[N // 3]
    h = to_host(P.arnoldi_bmgs(V, j, to_dev(w0), torch.zeros((j + 2) * 4, dtype=torch.float64, device="cuda")))
    assert (np.isnan(h[0]) if np.isnan(bad) else h[0] == bad * np.sign(v0)), h
    assert not np.isfinite(h).any()


@pytest.mark.parametrize("form", ["I", "sigma"])
def test_gmres_blocks_of_eight(form):
    """One long GMRES cycle (every block of 8 and each last-block size before
    it) gives the least-squares residual of the Krylov space: the estimate it
    stops on and the true residual agree."""
    at = W.paper(60, 8, 11, freq_norm=0)
    P = problem(at) if form == "I" else __import__("paper_2110_11873_gb300").Problem(at, form="sigma")
    b = P.rhs()
    for m in (1, 7, 8, 9, 16, 23, 40):
        x, info = P.solve(b, "gmres", restart=m, maxit=m, precond="none", rtol=1e-13)
        r = b - P.apply(x)
        rel = float(torch.linalg.vector_norm(r) / torch.linalg.vector_norm(b))
        assert abs(rel - info.err_est) <= 1e-11 + 1e-8 * info.err_est, (m, rel, info)


def _basis(N, j, rng):
    Q = []
    for _ in range(j + 1):
        v = rng.standard_normal(N)
        for _ in range(2):
            for u in Q:
                v = v - np.dot(u, v) * u
        Q.append(v / np.linalg.norm(v))
    return Q


def _normalised(P, N, j, Q, w0):
    """h_{j+1} and v_{j+1} of one step against the w that the step left."""
    gram = np.zeros((j + 2, 4))
    for i in range(1, j + 1):
        for d in range(1, min(i, 3) + 1):
            gram[i, d] = Q[i] @ Q[i - d]
    Vd = torch.zeros((j + 2) * N, dtype=torch.float64, device="cuda")
    Vd[: (j + 1) * N] = to_dev(np.concatenate(Q))
    wd = to_dev(w0)
    h = to_host(P.arnoldi_bmgs(Vd, j, wd, to_dev(gram.reshape(-1))))
    P.check()
    w = to_host(wd)
    big = np.abs(w).max()
    left = big * np.linalg.norm(w / big)   # |w| without underflow of its square
    v = to_host(Vd)[(j + 1) * N:]
    return h[-1] / left - 1.0, np.linalg.norm(v) - 1.0


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-8, 1e-12, 1e-18, 1e-100])
@pytest.mark.parametrize("j", range(8))
def test_pass_norm_of_small_w(scale, j):
    """h_{j+1} and v_{j+1} have the accuracy of FP64 relative to what is left of
    w, whatever its size beside the unit basis.  Both sides sum N squares in
    trees and chains of length < 1000: 1e-13 of the sum, half of it of its root;
    the scaling of v adds three roundings."""
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    rng = np.random.default_rng(j)
    Q = _basis(P.N, j, rng)
    dh, dv = _normalised(P, P.N, j, Q, scale * rng.standard_normal(P.N))
    assert abs(dh) < 2e-13 and abs(dv) < 2e-13, (dh, dv)


@pytest.mark.parametrize("left", [1e-6, 1e-10, 1e-14])
@pytest.mark.parametrize("j", [0, 2, 5])
def test_pass_norm_of_a_dependent_w(left, j):
    """A w almost in the span of the basis: the same for what is left of it."""
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    rng = np.random.default_rng(10 + j)
    Q = _basis(P.N, j, rng)
    r = rng.standard_normal(P.N)
    w0 = sum(c * q for c, q in zip(rng.standard_normal(j + 1), Q)) + left * r / np.linalg.norm(r)
    dh, dv = _normalised(P, P.N, j, Q, w0)
    assert abs(dh) < 2e-13 and abs(dv) < 2e-13, (dh, dv)


def test_a_copy_that_does_not_arrive_reports_timeout_and_the_problem_recovers():
    """Failure path of the streamed passes' bounded waits, without a device
    fault: in an armed step one CTA goes on without its copies (they land
    before it ends).  The next check reports RT_ETIMEOUT once; later steps are
    right again.  A step in the register kernels (8-byte aligned operands) takes
    no armed injection."""
    from paper_2110_11873_gb300 import _native as N

    for Ns, Nmu, Nnu in ((70, 16, 21), (300, 32, 101)):   # one tile per CTA; more tiles than stages
        P = problem(W.slab(Ns, Nmu, Nnu, 1e-4, 1e6, 6.0))
        V = torch.zeros(3 * P.N + 2, dtype=torch.float64, device="cuda")
        gram = torch.zeros(12, dtype=torch.float64, device="cuda")
        for armed in (1, 2):
            P.inject_wait_timeout(armed)
            for _ in range(armed):
                P.arnoldi_bmgs(V, 0, torch.ones(P.N, dtype=torch.float64, device="cuda"), gram)
            with pytest.raises(N.RTError) as ei:
                P.check()
            assert ei.value.status == N.RT_ETIMEOUT
            P.check()   # the condition was cleared by the check that reported it
            _step(P, P.N, 2, "normal", seed=armed)
        P.inject_wait_timeout(1)
        _step(P, P.N, 2, "normal", offset=1)
        P.inject_wait_timeout(0)


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_pass_digits_round_without_a_sign(sign):
    """Entries of one sign beside large ones that the basis vector does not
    meet (2^20, one to every 32 elements): the fixed-point unit is 2^-34 (two
    bits of headroom, 54 below), each entry of 1..2 is rounded to it, and the
    rounding errors average out: 0.29 units each, 0.29 * 2^-34 / sqrt(N) / 1.5
    of the dot on the mean, 4.4e-14 for N = 65,600; six times that is allowed.
    An eighth of a unit in one direction would be 5e-12."""
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    N = P.N
    rng = np.random.default_rng(5)
    w0 = sign * rng.uniform(1.0, 2.0, N)
    v = rng.uniform(0.5, 1.0, N)
    w0[::32] = 2.0 ** 20
    v[::32] = 0.0
    v /= np.linalg.norm(v)
    V = torch.zeros(5 * N, dtype=torch.float64, device="cuda")   # a step that forms the first dot on the integer pipe
    V[:N] = to_dev(v)
    h = to_host(P.arnoldi_bmgs(V, 3, to_dev(w0), torch.zeros(20, dtype=torch.float64, device="cuda")))
    exact = float(np.sum(w0.astype(np.longdouble) * v.astype(np.longdouble)))
    assert abs(h[0] / exact - 1.0) < 2.7e-13, h[0] / exact - 1.0


@pytest.mark.parametrize("scale", [1e-290, 1e-300, 1e-306])
@pytest.mark.parametrize("j", [0, 2, 3, 9])
def test_pass_of_a_w_near_the_smallest_numbers(scale, j):
    """Entries below 2^-961, where the fixed-point scales end: the coefficients
    and what is left of w keep the accuracy of the other cases, 1e-12 and 1e-11
    of |w| (the products with the basis round to multiples of 5e-324, 65,600 of
    them to 2e-319 at most)."""
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    N = P.N
    rng = np.random.default_rng(j)
    Q = _basis(N, j, rng)
    u0 = rng.standard_normal(N)
    gram = np.zeros((j + 2, 4))
    for i in range(1, j + 1):
        for d in range(1, min(i, 3) + 1):
            gram[i, d] = Q[i] @ Q[i - d]
    V = torch.zeros((j + 2) * N, dtype=torch.float64, device="cuda")
    V[: (j + 1) * N] = to_dev(np.concatenate(Q))
    wd = to_dev(scale * u0)
    h = to_host(P.arnoldi_bmgs(V, j, wd, to_dev(gram.reshape(-1))))
    P.check()
    href, w = _mgs(Q, u0)
    s = np.linalg.norm(u0)
    np.testing.assert_allclose(h[: j + 1] / scale, href[: j + 1], rtol=0, atol=1e-12 * s)
    np.testing.assert_allclose(to_host(wd) / scale, w, rtol=0, atol=1e-11 * s)


def test_pass_of_large_vectors_and_a_small_w():
    """A dot whose factors are far apart but whose value is ordinary: 1e300 and
    1e-300 (the basis of a caller need not be normalised for it)."""
    P = problem(W.slab(100, 8, 41, 1e-4, 1e6, 6.0))
    N = P.N
    rng = np.random.default_rng(2)
    v, w0 = rng.standard_normal(N), rng.standard_normal(N)
    V = torch.zeros(5 * N, dtype=torch.float64, device="cuda")
    V[:N] = to_dev(1e300 * v)
    h = to_host(P.arnoldi_bmgs(V, 3, to_dev(1e-300 * w0), torch.zeros(20, dtype=torch.float64, device="cuda")))
    assert abs(h[0] - v @ w0) < 1e-12 * np.linalg.norm(v) * np.linalg.norm(w0), h[0]


@pytest.mark.parametrize("scale", [1.0, 1e-300])
def test_pass_of_zero_tiles_before_others(scale):
    """Every other tile of w, or of the basis vectors, is zero: a warp that meets
    the zeros first takes no scale from them."""
    P = problem(W.slab(300, 32, 32, 1e-4, 1e6, 6.0))   # 2400 tiles, 8 to a CTA
    N, j = P.N, 6
    rng = np.random.default_rng(1)
    zero = np.arange(N) // 256 % 2 == 0
    u0 = np.where(zero, 0.0, rng.standard_normal(N))
    Q = np.where(zero[None] == (np.arange(j + 1) % 3 == 2)[:, None], rng.standard_normal((j + 1, N)), 0.0) / np.sqrt(N / 2)
    V = torch.zeros((j + 2) * N, dtype=torch.float64, device="cuda")
    V[: (j + 1) * N] = to_dev(Q.reshape(-1))
    gram = np.zeros((j + 2, 4))
    for i in range(1, j + 1):
        for d in range(1, min(i, 3) + 1):
            gram[i, d] = Q[i] @ Q[i - d]
    h = to_host(P.arnoldi_bmgs(V, j, to_dev(scale * u0), to_dev(gram.reshape(-1))))
    P.check()
    href, w = _mgs(Q, u0)
    np.testing.assert_allclose(h[: j + 1] / scale, href[: j + 1], rtol=0, atol=1e-12 * np.linalg.norm(u0))

@pytest.mark.parametrize("Nnu", [95, 152, 153, 456, 607, 608, 609])
def test_pass_grid_around_one_cta_per_sm(Nnu):
    """Vectors of 95 to 609 tiles: fewer than one per SM, one, and up to and past
    the length from which two CTAs share an SM."""
    P = problem(W.slab(8, 8, Nnu * 2, 1e-4, 1e6, 6.0))   # N = 256 * Nnu
    assert P.N == 256 * Nnu
    _step(P, P.N, 6, "normal", seed=Nnu)
