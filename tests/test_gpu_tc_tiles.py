"""Tensor-core boundary products at the edges of their 32- and 64-column tiles and of the
128-row tiles, against the FP32 products, to the tolerance of the other tensor-core tests."""
import numpy as np
import pytest

import paper_1309_5796_gb300 as lbm
from synth.inputs import A_JM, JS_T, K1_JM3, m_random_sphere

pytestmark = pytest.mark.gpu


# 8 to 1016 surface nodes; 2, 31 to 33, 63 and 64 instances
@pytest.mark.parametrize("n,B", [(1, 2), (4, 31), (5, 32), (6, 33), (11, 32), (13, 63), (12, 64)])
def test_tiles(n, B):
    from paper_1309_5796_gb300 import build
    build.build()
    with lbm.Context(0) as ctx:
        mesh = ctx.mesh_cube(2e-9, n)
        m = np.stack([m_random_sphere((n + 1) ** 3, 10 * n + b) for b in range(B)])
        out = []
        for prec in (lbm.LBM_MIXED, lbm.LBM_MIXED_TC):
            inst = ctx.instance_create(mesh, B, prec)
            inst.set_material(JS_T, A_JM, K1_JM3, [0.0, 0.1, 1.0])
            inst.set_field([0.1, 0.0, -1.0])
            inst.set_m(m)
            out.append(inst.evaluate(lbm.default_opts(lbm.LBM_MIXED)))
            inst.destroy()
        ctx.mesh_destroy(mesh)
    (ra, ha, ua), (rt, ht, ut) = out
    assert np.abs(ht - ha).max() <= 2e-5 * np.abs(ha).max()
    for x, y in zip(ra, rt):
        assert abs(x["energy"][4] - y["energy"][4]) <= 2e-5 * (abs(x["energy"][4]) + 1e-20)
