"""The FP64 operator on large problems with a profile symmetric on the
frequency grid (rays p and Nnu-1-p solved together) against the oracle and
against the general kernels.

The general kernels run on the same atmosphere when the profile is passed in
with one frequency moved by two units in the last place: the two problems then
differ by 1e-16 of the operator, far below the tolerance.  Forms covered: odd
and even Nnu, lane groups that end inside a warp, the formal solvers with two
step terms, every apply mode (plain, right-hand side, local-Lambda and Jacobi
inside GMRES, with and without the fused normalisation)."""
import numpy as np
import pytest
import torch

import rt_workloads as W
from oracle.transfer import Transfer
from paper_2110_11873_gb300 import Problem
from gpu_util import assert_close_scaled, problem, to_dev, to_host

pytestmark = pytest.mark.gpu

# N = 2 Ns Nmu Nnu just above the size from which the pairs are taken (4 Mi)
SHAPES = [(130, 64, 253), (700, 30, 100), (53, 200, 201)]


def _atm(shape, fs):
    at = W.slab(*shape, 1e-4, 1e8, 8.0, eps=1e-3, Bc=0.3, formal_solver=fs)
    assert at.N >= 4 << 20
    return at


def _general(at):
    """The same atmosphere through the general kernels."""
    g = problem(at).grids()
    phi = g["phi"].copy()
    phi[3] = np.nextafter(np.nextafter(phi[3], 1.0), 1.0)
    centre = g["phi"][0] / g["phi_hat"][0]   # line-centre scaling: phi_hat = phi / phi(0)
    return Problem(at, phi=phi, phi_center=float(centre))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("fs", [W.FS_DELO_LINEAR, W.FS_IMPLICIT_EULER, W.FS_TRAPEZOIDAL])
def test_pairs_against_the_general_kernels(shape, fs):
    at = _atm(shape, fs)
    P, G = problem(at), _general(at)
    x = to_dev(W.random_vector(at.N, 5))
    assert_close_scaled(to_host(P.apply(x)), to_host(G.apply(x)), 1e-12)
    b, bg = P.rhs(), G.rhs()
    assert_close_scaled(to_host(b), to_host(bg), 1e-12)
    assert_close_scaled(to_host(P.precond_local_lambda(x)), to_host(G.precond_local_lambda(x)), 1e-12)
    for prec in ("none", "jacobi", "local_lambda"):
        kw = dict(restart=6, maxit=6, precond=prec, rtol=1e-14)
        y, _ = P.solve(b, "gmres", **kw)
        yg, _ = G.solve(bg, "gmres", **kw)
        assert_close_scaled(to_host(y), to_host(yg), 1e-10)


def test_pairs_against_the_oracle():
    at = _atm(SHAPES[0], W.FS_DELO_LINEAR)
    P, tr = problem(at), Transfer(at)
    x = W.random_vector(at.N, 6)
    assert_close_scaled(to_host(P.apply(to_dev(x))), tr.apply_I(x), 1e-10)
    assert_close_scaled(to_host(P.rhs()), tr.rhs_I(), 1e-10)
    assert_close_scaled(to_host(P.jacobi_diag()), tr.jacobi_I(), 1e-10)


@pytest.mark.parametrize("x_max,Nnu", [(8.0, 201), (6.0, 100), (4.0, 57)])
def test_grids_do_not_depend_on_the_kernels(x_max, Nnu):
    """The same frequencies, profile and weights to the bit on both sides of the
    size from which pairs are solved together; above it a symmetric x gives a
    symmetric A x to the bit, which only the pairs do (x_p = x_min + p h rounds
    differently in the two halves)."""
    Ns = (4 << 20) // (2 * 64 * Nnu)
    small, large = (problem(W.slab(n, 64, Nnu, 1e-4, 1e8, x_max)) for n in (Ns - 8, Ns + 8))
    assert small.N < 4 << 20 <= large.N
    a, b = small.grids(), large.grids()
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    x = to_dev(W.random_vector(large.N, 7)).reshape(-1, Nnu)
    x = x + x.flip(1)
    y = large.apply(x.reshape(-1)).reshape(-1, Nnu)
    assert torch.equal(y, y.flip(1))
