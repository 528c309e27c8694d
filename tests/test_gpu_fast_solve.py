"""Potential solves on Kuhn cubes by fast diagonalisation (csrc/fast_solve.cu)
against the diagonally preconditioned CG of the grid-wide kernel
(lbm_solve_opts.pcg_kernel = 1).

Both solve to a relative residual of 1e-13 (FP64), 1e-10 (FP64 iterated in
FP32) or 1e-6 (FP32).  The smallest nonzero eigenvalue of the stiffness over its
largest is about 1/n^2 (1/7744 at n = 88), so the potentials agree to that
factor times the residual: 1e-9, 1e-6 with the FP32 iterations, and in FP32 (a
smooth right-hand side, whose error the residual bounds far more closely) to the
2e-5 that the FP32 parity tests use.
"""
import numpy as np
import pytest

import paper_1309_5796_gb300 as lbm
from synth.inputs import A_JM, JS_T, K1_JM3, tilted_axis

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1309_5796_gb300 import build
    build.build()
    c = lbm.Context(0)
    yield c
    c.close()


def _m(n, B, seed):
    rng = np.random.default_rng(seed)
    g = np.arange(n + 1) / n
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    p = np.stack([x.ravel(), y.ravel(), z.ravel()], 1)
    m = np.stack([np.stack([np.sin(2 * p[:, 0] + 0.3 * b), np.cos(1.5 * p[:, 1] - b), 0.5 + p[:, 2]], 1) for b in range(B)])
    m += 0.05 * rng.standard_normal(m.shape)
    return m / np.linalg.norm(m, axis=-1, keepdims=True)


def _run(ctx, mesh, n, B, prec, m, **opts):
    inst = ctx.instance_create(mesh, B, prec)
    inst.set_material(JS_T, A_JM, K1_JM3, tilted_axis(3.0, 0.4))
    inst.set_field(np.array([0.1, 0.0, -2.0]))
    inst.set_m(m)
    res, h, u = inst.evaluate(lbm.default_opts(prec, **opts))
    inst.destroy()
    return res, h, u


# smallest cubes, both parities of n, halves that fill and miss a tile of 4, one to
# several planes per CTA, widths 1, 2 and 4, planes in global memory (66 FP64, 88 FP32)
CASES = [(1, 1, 0), (1, 4, 1), (2, 1, 0), (2, 3, 1), (3, 2, 0), (4, 4, 1), (5, 1, 1), (6, 5, 0), (7, 8, 1), (8, 2, 0),
         (13, 3, 1), (14, 6, 0), (15, 1, 0), (16, 16, 1), (17, 1, 0), (31, 4, 1), (33, 1, 0), (66, 1, 0), (88, 1, 1)]


@pytest.mark.parametrize("n,B,prec", CASES)
def test_fast_solve_matches_cg(ctx, n, B, prec):
    mesh = ctx.mesh_cube(2e-9, n)
    m = _m(n, B, 7 * n + B)
    variants = [dict()] if prec else [dict(), dict(cg_mixed_iter=1, cg_tol=1e-10)]
    ref = _run(ctx, mesh, n, B, prec, m, pcg_kernel=1)
    for v in variants:
        tol = 2e-5 if prec else (1e-6 if v else 1e-9)
        res, h, u = _run(ctx, mesh, n, B, prec, m, **v)
        for b in range(B):
            assert np.linalg.norm(u[b] - ref[2][b]) <= tol * np.linalg.norm(ref[2][b]), (b, v)
            assert np.linalg.norm(h[b] - ref[1][b]) <= tol * np.linalg.norm(ref[1][b]), (b, v)
            if not prec and not v:
                # two Neumann solves of one pair of steps each, two Dirichlet solves of one step
                assert res[b]["cg_iters1"] <= 6 and res[b]["cg_iters2"] <= 4
    ctx.mesh_destroy(mesh)


@pytest.mark.parametrize("n", [5, 12, 21])
@pytest.mark.parametrize("prec", [0, 1])
def test_bits_do_not_depend_on_the_batch(ctx, n, prec):
    """An instance's first-stage potential has the same bits in every batch (other
    widths, cluster sizes and thread counts); the second stage follows the boundary
    product, whose summation order does depend on the batch."""
    mesh = ctx.mesh_cube(2e-9, n)
    m = _m(n, 12, 3)
    u = {B: _run(ctx, mesh, n, B, prec, m[:B])[2][:, 0] for B in (1, 2, 3, 12)}
    for B in (2, 3, 12):
        assert np.array_equal(u[B][0], u[1][0])
    assert np.array_equal(u[12][:3], u[3])
    ctx.mesh_destroy(mesh)


@pytest.mark.parametrize("n,B", [(8, 192), (14, 192), (20, 128)])
def test_a_converged_system_waits(ctx, n, B):
    """Tolerances near and below FP32's rounding, where the systems that share a cluster
    (two do at these sizes) need different numbers of pairs of steps: one that has
    converged takes no further step, so every instance's first-stage potential has the
    bits it has alone."""
    mesh = ctx.mesh_cube(2e-9, n)
    m = _m(n, B, 11)
    rng = np.random.default_rng(5)
    m[1::4] = rng.standard_normal(m[1::4].shape)   # rough right-hand sides beside smooth ones
    m[2::4, :, :2] *= 0.02
    m /= np.linalg.norm(m, axis=-1, keepdims=True)
    mixed = 0
    for tol in (1e-7, 7e-8, 5e-8, 4e-8, 3e-8, 2e-8, 1e-8, 1e-13):
        counts = set()
        u = _run(ctx, mesh, n, B, 1, m, cg_tol=tol)[2]
        for b in (*range(12), B // 2, B - 1):
            res, _, one = _run(ctx, mesh, n, 1, 1, m[b:b + 1], cg_tol=tol)
            counts.add(res[0]["cg_iters1"])
            assert np.array_equal(u[b, 0], one[0, 0]), (tol, b)
        mixed += len(counts) > 1
    assert mixed   # some instances did take more steps than others
    ctx.mesh_destroy(mesh)


@pytest.mark.parametrize("n,prec,opts,tol", [
    (82, 0, dict(cg_mixed_iter=1, cg_tol=1e-10), 1e-6), (96, 1, dict(), 2e-5)])
def test_the_largest_cubes(ctx, n, prec, opts, tol):
    """FP64 solves iterated in FP32 with their planes in global memory, and the largest
    cube there is."""
    mesh = ctx.mesh_cube(2e-9, n)
    m = _m(n, 1, 5)
    _, h, u = _run(ctx, mesh, n, 1, prec, m, **opts)
    _, hr, ur = _run(ctx, mesh, n, 1, prec, m, pcg_kernel=1, **opts)
    ctx.mesh_destroy(mesh)
    assert np.linalg.norm(u - ur) <= tol * np.linalg.norm(ur)
    assert np.linalg.norm(h - hr) <= tol * np.linalg.norm(hr)
