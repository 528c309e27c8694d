"""The node kernels (right-hand side, field and energies, step control, trial point):
their lanes go to the instances that still run, in blocks sized by the work."""
import numpy as np
import pytest

import paper_1309_5796_gb300 as lbm
from synth.inputs import A_JM, JS_T, K1_JM3, m_perturbed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1309_5796_gb300 import build
    build.build()
    c = lbm.Context(0)
    yield c
    c.close()


def _instance(ctx, mesh, m, prec, field):
    inst = ctx.instance_create(mesh, len(m), prec)
    inst.set_material(JS_T, A_JM, K1_JM3, [0.05, 0.0, 1.0])
    inst.set_field(np.tile(field, (len(m), 1)))
    inst.set_m(m)
    return inst


@pytest.mark.parametrize("n,B", [(2, 1), (2, 256), (3, 129), (7, 64), (7, 65), (9, 3), (9, 32), (9, 33), (10, 4)])
def test_batch_matches_single(ctx, n, B):
    """Every instance of a batch has the values it has alone.  FP64: the sums differ in
    order only, N eps (under 1e-12 at these sizes) of the quantities' scales, and the
    boundary products by some 1e-13."""
    mesh, N = ctx.mesh_cube(2e-9, n), (n + 1) ** 3
    m = np.stack([m_perturbed(N, 70 + b, 0.3, (0.2, 0.1 * (b % 7), 1.0)) for b in range(B)])
    inst = _instance(ctx, mesh, m, lbm.LBM_FP64, [0.1, 0.0, -0.7])
    res, h, u = inst.evaluate(lbm.default_opts(lbm.LBM_FP64))
    inst.destroy()
    for b in sorted({0, B // 2, B - 1}):
        one = _instance(ctx, mesh, m[b:b + 1], lbm.LBM_FP64, [0.1, 0.0, -0.7])
        r1, h1, u1 = one.evaluate(lbm.default_opts(lbm.LBM_FP64))
        one.destroy()
        scale = np.abs(r1[0]["energy"]).max()
        assert np.abs(np.array(res[b]["energy"]) - r1[0]["energy"]).max() <= 1e-11 * scale
        for q in ("torque", "gg"):
            assert abs(res[b][q] - r1[0][q]) <= 1e-10 * abs(r1[0][q])
        assert np.abs(np.reshape(h, (B, N, 3))[b] - np.reshape(h1, (N, 3))).max() <= 1e-11 * np.abs(h1).max()
    ctx.mesh_destroy(mesh)


def test_bits_do_not_depend_on_who_has_finished(ctx):
    """An instance minimises to the same bits beside instances that run as long and beside
    ones that stop at once."""
    n, B, prec = 6, 8, lbm.LBM_FP64
    mesh, N = ctx.mesh_cube(2e-9, n), (n + 1) ** 3
    m = np.stack([m_perturbed(N, 90 + b, 0.3, (0.3, 0.05 * b, 1.0)) for b in range(B)])
    inst = _instance(ctx, mesh, m, prec, [0.0, 0.0, -0.5])
    res = inst.minimise(lbm.default_opts(prec))
    relaxed = np.reshape(inst.get_m(), (B, N, 3)).copy()
    inst.destroy()
    k = int(np.argmax([r["evaluations"] for r in res]))
    mixed = relaxed.copy()
    mixed[k] = m[k]
    inst = _instance(ctx, mesh, mixed, prec, [0.0, 0.0, -0.5])
    res2 = inst.minimise(lbm.default_opts(prec))
    again = np.reshape(inst.get_m(), (B, N, 3))
    inst.destroy()
    ctx.mesh_destroy(mesh)
    assert min(r["evaluations"] for r in res2) < res2[k]["evaluations"]
    assert res2[k]["evaluations"] == res[k]["evaluations"]
    assert np.array_equal(again[k], relaxed[k])


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_MIXED])
def test_no_easy_axis_no_anisotropy(ctx, prec):
    """A material without an easy axis (0, 0, 0) has no anisotropy energy and no anisotropy
    field, whatever its K1, beside an instance with an axis (whose energy is the sum of
    K1 V |m x a|^2: every term of it is positive here)."""
    n, B = 5, 2
    mesh, N = ctx.mesh_cube(2e-9, n), (n + 1) ** 3
    m = np.stack([m_perturbed(N, 31 + b, 0.3, (0.4, 0.1, 1.0)) for b in range(B)])
    out = {}
    for k1 in (K1_JM3, 0.0):
        inst = ctx.instance_create(mesh, B, prec)
        inst.set_material(JS_T, A_JM, k1, [[0.0, 0.0, 0.0], [0.0, 0.0, 1.0]])
        inst.set_field(np.array([0.1, 0.0, -0.7]))
        inst.set_m(m)
        out[k1] = inst.evaluate(lbm.default_opts(prec))
        inst.destroy()
    (res, h, _), (plain, h0, _) = out[K1_JM3], out[0.0]
    assert res[0]["energy"] == plain[0]["energy"] and np.array_equal(h[0], h0[0])
    assert res[0]["energy"][1] == 0.0 < res[1]["energy"][1]
    if prec == lbm.LBM_FP64:   # the entry point that allocates nothing
        torch = pytest.importorskip("torch")
        d_m = torch.from_numpy(m[0]).to("cuda")
        d_e = torch.zeros(5, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.evaluate_noalloc(mesh, JS_T, A_JM, K1_JM3, [0.0, 0.0, 0.0], np.array([0.1, 0.0, -0.7]), d_m.data_ptr(),
                             d_energy=d_e.data_ptr())
        torch.cuda.synchronize()
        assert float(d_e[1]) == 0.0 and float(d_e[0]) > 0.0
    ctx.mesh_destroy(mesh)
