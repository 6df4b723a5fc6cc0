"""Restart cycles of GMRES launched as several graphs.

Cycle lengths and iteration limits below, at and past the graphs' 8 steps and
the longest last graph (12 steps), and stops by the tolerance at each of those places
of a longer cycle: iteration and restart counts and iterates against the oracle.
A stop at the end of a graph is found by the first kernel of the next one, one
inside it leaves the rest of the cycle unlaunched.  Sigma-form vectors of more
than 1024 values take the streamed block passes with the normalisation in a kernel
of its own."""
import numpy as np
import pytest

import rt_workloads as W
from oracle import krylov as K
from oracle.transfer import Transfer
from paper_2110_11873_gb300 import Problem
from paper_2110_11873_gb300 import _native as N

from gpu_util import assert_iterate, perturbed, problem, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    at = W.slab(24, 8, 11, 1e-4, 1e6, 6.0)
    tr = Transfer(at)
    return problem(at), tr, tr.rhs_I()


@pytest.mark.parametrize("restart,maxit", [(30, 8), (30, 9), (30, 16), (30, 24), (30, 38), (1, 4), (5, 23), (8, 17),
                                           (12, 12), (12, 25), (13, 13), (13, 30), (20, 20), (20, 29), (21, 50),
                                           (160, 40)])
def test_iteration_limits_around_the_segments(small, restart, maxit):
    P, tr, b = small
    d = tr.jacobi_I()
    kw = dict(M_inv=lambda v: v / d, restart=restart, tol=1e-30, maxit=maxit)
    xg, info = P.solve(to_dev(b), "gmres", restart=restart, precond="jacobi", rtol=1e-30, maxit=maxit)
    assert info.status == N.RT_ENOTCONV and info.iters == maxit
    assert info.restarts == -(-maxit // restart)
    xo, io = K.gmres(tr.apply_I, b, **kw)
    assert io.iters == maxit
    xp, _ = K.gmres(tr.apply_I, perturbed(b, 1), **kw)
    assert_iterate(to_host(xg), xo, xp, f"gmres({restart}) after {maxit}")


@pytest.mark.parametrize("steps", [1, 7, 8, 9, 15, 16, 17, 23, 24, 25, 29])
@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_stops_by_tolerance_around_the_segments(small, steps, precision):
    """The tolerance lies between the estimates of steps - 1 and steps."""
    P, tr, b = small
    _, full = P.solve(to_dev(b), "gmres", restart=30, precond="jacobi", rtol=1e-30, maxit=30, hist_cap=64)
    est = np.concatenate([[1.0], full.history])
    assert est.size == 31
    rtol = float(np.sqrt(est[steps - 1] * est[steps]))
    x, info = P.solve(to_dev(b), "gmres", restart=30, precond="jacobi", rtol=rtol, maxit=30, precision=precision)
    if precision == "fp64":
        assert info.status == N.RT_OK and info.iters == steps and info.restarts == 1, (rtol, info)
    r = b - tr.apply_I(to_host(x))
    if info.status == N.RT_OK:
        assert np.linalg.norm(r) / np.linalg.norm(b) < rtol
    assert abs(np.linalg.norm(r) / np.linalg.norm(b) - info.rel_resid) < 1e-10


def test_sigma_form_of_more_than_1024_values():
    """The estimate that a cycle of m steps ends with and the true residual agree."""
    at = W.paper(600, 8, 11, freq_norm=0)
    P = Problem(at, form="sigma")
    b = P.rhs()
    for m in (1, 7, 8, 9, 16, 23, 40):
        x, info = P.solve(b, "gmres", restart=m, maxit=m, precond="none", rtol=1e-13)
        rel = float((b - P.apply(x)).norm() / b.norm())
        assert abs(rel - info.err_est) <= 1e-11 + 1e-8 * info.err_est, (m, rel, info)
