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


def test_no_room_for_sums_that_no_product_takes():
    """A batch whose boundary products run on the tensor cores holds their scratch and not
    the partial sums of the other batched product as well (8 splits x nb x 2B doubles here,
    44 MB; two words of each vector and 8 splits x nb x B x 2 FP32 sums, 28 MB)."""
    from paper_1309_5796_gb300 import build
    build.build()
    torch = pytest.importorskip("torch")
    with lbm.Context(0) as ctx:
        mesh = ctx.mesh_cube(2e-9, 30)
        used = {}
        for prec in (lbm.LBM_MIXED_TC, lbm.LBM_MIXED, lbm.LBM_MIXED_TC):   # the first brings the mesh's padded copies
            f0 = torch.cuda.mem_get_info()[0]
            inst = ctx.instance_create(mesh, 64, prec)
            used[prec] = f0 - torch.cuda.mem_get_info()[0]
            inst.destroy()
        ctx.mesh_destroy(mesh)
    assert 0 < used[lbm.LBM_MIXED_TC] <= used[lbm.LBM_MIXED] - (10 << 20)
