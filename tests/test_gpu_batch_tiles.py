"""The batch's tiled FP32 formal solver, and admission under a small budget.

Depths at which the number of depth tiles and the last tile's length change
(one tile, a tile more per 8 steps, all 8 tiles with and without a short last
one), ray groups that end inside a warp, the three formal solvers, all resident
together: every solution that the oracle's GMRES(10) finds has the residual
asked for with the oracle's FP64 operator and agrees with the FP64 single-instance solver's.

Tolerances: the residual is the stopping rule's, 1e-9, with the oracle's own
rounding on top (1e-12); two solutions of residual 1e-9 differ by at most
2e-9 |A^-1| |b|, and |A^-1| <= 1/eps = 100 here, hence 2e-7 |b|, with |x| >= |b|/2
(|A| < 2)."""
import time

import numpy as np
import pytest

import rt_workloads as W
from oracle import krylov as K
from oracle.transfer import Transfer
from paper_2110_11873_gb300 import Server
from paper_2110_11873_gb300 import _native as N
from gpu_util import problem, to_host

pytestmark = pytest.mark.gpu


def _drain(srv, tickets):
    out, t0 = {}, time.time()
    while len(out) < len(tickets):
        for t in tickets:
            if t not in out:
                r = srv.poll(t)
                if r is not None:
                    out[t] = r
        assert time.time() - t0 < 120
    return [out[t] for t in tickets]


def _atms(fs):
    return [W.slab(Ns, Nmu, Nnu, 1e-4, 1e6, 6.0, eps=1e-2, Bc=0.2, formal_solver=fs)
            for Ns, Nmu, Nnu in [(2, 4, 5), (9, 4, 7), (17, 6, 11), (40, 4, 33), (65, 8, 21), (66, 2, 3), (130, 4, 9)]]


@pytest.mark.parametrize("fs", [W.FS_DELO_LINEAR, W.FS_IMPLICIT_EULER, W.FS_TRAPEZOIDAL])
@pytest.mark.parametrize("precond", ["local_lambda", "jacobi", "none"])
def test_tiled_batch_solves(fs, precond):
    atms = _atms(fs)
    srv = Server(mem_budget_bytes=1 << 30, max_slots=16, restart=10, precond=precond, precision="fp32_refine")
    try:
        got = _drain(srv, [srv.submit(a, rtol=1e-9) for a in atms])
    finally:
        srv.close()
    for a, (st, info, x) in zip(atms, got):
        tr = Transfer(a)
        b = tr.rhs_I()
        d = tr.jacobi_I()
        Minv = {"none": None, "jacobi": lambda v: v / d, "local_lambda": tr.local_lambda_I_inverse}[precond]
        xo, _ = K.gmres(tr.apply_I, b, M_inv=Minv, restart=10, tol=1e-9, maxit=600)
        stagnates = np.linalg.norm(b - tr.apply_I(xo)) > 1e-6 * np.linalg.norm(b)
        if st == N.RT_ENOTCONV and stagnates:   # 2 x 3 rays: GMRES(10) stagnates in the oracle too
            continue
        assert st == 0, (a.Ns, info)
        assert np.linalg.norm(b - tr.apply_I(x)) <= (1e-9 + 1e-12) * np.linalg.norm(b)
        P = problem(a)
        xs, one = P.solve(P.rhs(), "gmres", restart=10, precond="local_lambda", rtol=1e-9)
        assert one.ok
        assert np.linalg.norm(x - to_host(xs)) <= 4e-7 * np.linalg.norm(x)


def test_requests_wait_for_the_memory_of_retiring_ones():
    """A budget that holds one instance at a time: every request is admitted
    as the one before it has been copied out, none fails for lack of memory."""
    atms = [W.slab(60, 8, 21, 1e-4, 1e6, 6.0, eps=1e-2, Bc=0.1 * i) for i in range(6)]
    srv = Server(mem_budget_bytes=10 << 20, max_slots=4, restart=10, precision="fp32_refine")
    try:
        got = _drain(srv, [srv.submit(a, rtol=1e-9) for a in atms])
        assert srv.stats()["arena_in_use"] == 0
    finally:
        srv.close()
    assert [st for st, _, _ in got] == [0] * len(atms)
