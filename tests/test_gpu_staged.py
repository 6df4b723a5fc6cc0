"""The fast FP32 apply: vectorised quadrature and the formal solver with
tensor-copy staging of x (GPU).

Checked against the oracle's FP64 operator at 2e-5 relative to the largest
entry (the bound of every FP32 apply), and against the register-ring FP32
kernels (selected by RT_NO_TMA=1) at 1e-5: the two paths sum the quadrature
in different orders and split the depth scan into different tiles, so they
agree to FP32 rounding accumulated along the rays, not bit for bit.
Shapes cover partial ray groups (Nmu/2*Nnu not a multiple of 32), depth tiles
that end inside a stage, boxes that start below height 0 or end above Ns-1
(zero-filled rows), the minimal Ns = 2, the three formal solvers, a layout
the tensor copies cannot serve and an input that is not 16-byte aligned (the
register kernels run), and the FP32-REFINE solvers, whose FP64-vector applies
(no preconditioner, Jacobi, local Lambda) run inside captured graphs.  The
failure path of the bounded tensor-copy waits is driven by host-armed
injection (no device fault).
"""
import numpy as np
import pytest
import torch

import rt_workloads as W
from oracle.transfer import Transfer

from gpu_util import assert_close_scaled, problem, to_dev, to_host

pytestmark = pytest.mark.gpu

TOL32 = 2e-5
TOL_PATHS = 1e-5

SHAPES = [
    ("ragged-37x8x10", W.slab(37, 8, 10, 1e-4, 1e6, 6.0, Bc=0.3, eps=1e-3)),
    ("ns2-4x2", W.slab(2, 4, 2, 1e-2, 1e2, 3.0)),
    ("ns19-16x6-euler", W.slab(19, 16, 6, 1e-3, 1e4, 5.0, eps=1e-2).with_(formal_solver=W.FS_IMPLICIT_EULER)),
    ("ns53-8x12-trap", W.slab(53, 8, 12, 1e-3, 1e4, 5.0).with_(formal_solver=W.FS_TRAPEZOIDAL)),
    ("slab70", W.slab70()),
    ("paper-140", W.paper(140)),
    ("slab300", W.slab300()),
]


def _pair(at, monkeypatch):
    staged = problem(at)
    monkeypatch.setenv("RT_NO_TMA", "1")
    ring = problem(at)
    monkeypatch.delenv("RT_NO_TMA")
    assert staged.staged_formal and not ring.staged_formal
    return staged, ring


@pytest.mark.parametrize("name,at", SHAPES, ids=[s[0] for s in SHAPES])
def test_staged_apply_matches_the_oracle_and_the_register_path(name, at, monkeypatch):
    staged, ring = _pair(at, monkeypatch)
    tr = Transfer(at)
    x = W.random_vector(tr.N, 23)
    xd = to_dev(x, torch.float32)
    ys = staged.apply_f32(xd)
    yr = ring.apply_f32(xd)
    staged.check()
    ys_h = to_host(ys)
    assert_close_scaled(ys_h, tr.apply_I(x.astype(np.float32).astype(np.float64)), TOL32, name)
    assert_close_scaled(ys_h, to_host(yr), TOL_PATHS, name + " vs register path")


def test_deep_atmosphere_matches_the_register_path(monkeypatch):
    at = W.sweep(1000)
    staged, ring = _pair(at, monkeypatch)
    x = torch.rand(staged.N, device="cuda", dtype=torch.float32, generator=torch.Generator("cuda").manual_seed(5))
    ys = staged.apply_f32(x)
    yr = ring.apply_f32(x)
    staged.check()
    assert_close_scaled(to_host(ys), to_host(yr), TOL_PATHS, "sweep1000")


def test_layout_the_copies_cannot_serve_uses_the_register_kernels():
    at = W.slab(20, 4, 3, 1e-3, 1e3, 4.0)   # Nmu/2*Nnu = 6: ray groups not 16-byte aligned
    P = problem(at)
    assert not P.staged_formal
    tr = Transfer(at)
    x = W.random_vector(tr.N, 3)
    y = to_host(P.apply_f32(to_dev(x, torch.float32)))
    assert_close_scaled(y, tr.apply_I(x.astype(np.float32).astype(np.float64)), TOL32, "unaligned layout")


def test_unaligned_input_takes_the_register_kernels(monkeypatch):
    at = W.slab70()
    staged, ring = _pair(at, monkeypatch)
    buf = torch.rand(staged.N + 1, device="cuda", dtype=torch.float32, generator=torch.Generator("cuda").manual_seed(9))
    x = buf[1:]   # 4 bytes past a 16-byte boundary
    assert x.data_ptr() % 16 != 0
    assert torch.equal(staged.apply_f32(x), ring.apply_f32(x.clone()))
    staged.check()


@pytest.mark.parametrize("precond", ["none", "jacobi", "local_lambda"])
def test_fp32_refine_solves_through_the_staged_kernels(precond, monkeypatch):
    at = W.slab70()
    staged, ring = _pair(at, monkeypatch)
    tr = Transfer(at)
    b_h = tr.rhs_I()
    x_ex = tr.exact_I()
    b = to_dev(b_h)
    iters, refines = {}, {}
    for name, P in (("staged", staged), ("ring", ring)):
        x, res = P.solve(b, "gmres", restart=30, precond=precond, precision="fp32_refine", rtol=1e-8, maxit=20000,
                         inner_rtol=1e-4)
        assert res.status == 0, (name, res)
        xh = to_host(x)
        assert np.linalg.norm(b_h - tr.apply_I(xh)) / np.linalg.norm(b_h) < 1e-8, name
        if precond == "local_lambda":   # well conditioned: the residual bounds the error
            assert np.linalg.norm(xh - x_ex) / np.linalg.norm(x_ex) < 1e-6, name
        iters[name] = res.iters
        refines[name] = res.refine_steps
    # same algorithm, FP32 arithmetic in a different order.  Without a good
    # preconditioner the restarted iteration count reacts chaotically to
    # rounding (as the oracle's own counts do under 1e-15 perturbations), so
    # counts are compared only for the well-conditioned local-Lambda system:
    # every refinement step's inner solve stops where its FP32 residual
    # estimate crosses inner_rtol, which two FP32 operators reach within a
    # couple of Arnoldi steps of each other.
    if precond == "local_lambda":
        assert abs(iters["staged"] - iters["ring"]) <= 2 * (refines["ring"] + 1), (iters, refines)


def test_a_copy_wait_that_gives_up_reports_timeout_and_the_problem_recovers():
    """Failure path of the bounded tensor-copy waits, without a device fault:
    an armed apply treats one warp's first wait as given up (the warp flags
    the problem, waits for its copies in flight and skips its tile).  The
    next check reports RT_ETIMEOUT once; later applies are correct again."""
    from paper_2110_11873_gb300 import _native as N

    at = W.slab70()
    tr = Transfer(at)
    P = problem(at)
    assert P.staged_formal
    x = W.random_vector(tr.N, 4)
    xd = to_dev(x, torch.float32)
    ref = tr.apply_I(x.astype(np.float32).astype(np.float64))
    for armed in (1, 2):
        P.inject_wait_timeout(armed)
        for _ in range(armed):
            P.apply_f32(xd)
        with pytest.raises(N.RTError) as ei:
            P.check()
        assert ei.value.status == N.RT_ETIMEOUT
        P.check()   # the condition was cleared by the check that reported it
        y = to_host(P.apply_f32(xd))
        P.check()
        assert_close_scaled(y, ref, TOL32, f"after {armed} injected timeouts")
    with pytest.raises(N.RTError):
        P.inject_wait_timeout(-1)


def test_deep_atmosphere_with_few_rays_through_the_fused_normalisation():
    """N_s = 1001 with 40 rays per height: one quadrature column, so the
    fused-normalisation quadrature of GMRES takes several heights per CTA
    (one wave of resident CTAs) and its last CTA a ragged remainder.  The
    FP32-operator Jacobi-GMRES with FP64 refinement runs through it and
    meets the stopping rule with the oracle's FP64 operator; its solution
    agrees with the FP64 solver's within the refinement's accuracy."""
    at = W.slab(1001, 8, 5, 1e-4, 1e8, 6.0, eps=1e-2)
    tr = Transfer(at)
    P = problem(at)
    assert P.staged_formal
    b_h = tr.rhs_I()
    b = to_dev(b_h)
    x32, r32 = P.solve(b, "gmres", restart=30, precond="jacobi", precision="fp32_refine", rtol=1e-9, maxit=20000,
                       inner_rtol=1e-4)
    assert r32.status == 0 and r32.refine_steps >= 2, r32
    xh = to_host(x32)
    assert np.linalg.norm(b_h - tr.apply_I(xh)) / np.linalg.norm(b_h) < 1e-9
    x64, r64 = P.solve(b, "gmres", restart=30, precond="local_lambda", rtol=1e-11)
    assert r64.status == 0, r64
    assert_close_scaled(xh, to_host(x64), 1e-6, "fp32-refine vs fp64")


@pytest.mark.parametrize("name,at", [("slab300", W.slab300()), ("sweep500", W.sweep(500))])
def test_chained_applies_back_to_back_equal_synchronised_ones(name, at):
    """Each apply's output is the next one's input, eight in a row on one
    stream with no host synchronisation between them, FP32 (staged path)
    and FP64.  The kernels of an apply are programmatic dependents of the
    kernels before them, and the staged formal solver copies x before its
    own wait; the chain must give bit for bit what the same chain gives with
    a device synchronisation after every apply."""
    P = problem(at)
    assert P.staged_formal
    g = torch.Generator(device="cuda").manual_seed(11)
    for dt, fn in ((torch.float32, P.apply_f32), (torch.float64, P.apply)):
        x0 = torch.rand(P.N, dtype=dt, device="cuda", generator=g)
        bufs = [x0.clone()] + [torch.empty_like(x0) for _ in range(8)]
        for i in range(8):
            fn(bufs[i], out=bufs[i + 1])
        chained = to_host(bufs[8])
        ref = x0.clone()
        for _ in range(8):
            nxt = torch.empty_like(ref)
            fn(ref, out=nxt)
            torch.cuda.synchronize()
            ref = nxt
        P.check()
        np.testing.assert_array_equal(chained, to_host(ref), err_msg=f"{name} {dt}")


@pytest.mark.parametrize("Ns,Nmu,Nnu", [(5, 2, 2), (9, 2, 255), (9, 2, 256), (9, 2, 257), (7, 6, 171), (3, 30, 101), (456, 2, 3),
                                        (457, 2, 3), (3, 2, 1024), (3, 2, 1025), (460, 2, 511), (460, 2, 513)])
def test_register_path_ray_counts_around_the_quadrature_block(Ns, Nmu, Nnu, monkeypatch):
    """The flat FP32 quadrature with less than a warp of rays, and below, at and
    past one and two rounds of its threads and four rays of each, on few and on
    many heights."""
    at = W.slab(Ns, Nmu, Nnu, 1e-3, 1e4, 5.0, eps=1e-2)
    monkeypatch.setenv("RT_NO_TMA", "1")
    P = problem(at)
    tr = Transfer(at)
    x = W.random_vector(tr.N, 3)
    y = to_host(P.apply_f32(to_dev(x, torch.float32)))
    assert_close_scaled(y, tr.apply_I(x.astype(np.float32).astype(np.float64)), TOL32, f"{Ns} x {Nmu} x {Nnu}")
