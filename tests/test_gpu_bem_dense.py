"""Dense boundary products y = B x and y = B^T x: one instance in one pass over B, batches
in tiles of 8, 16 and 32 instances with split sums."""
import numpy as np
import pytest

import paper_1309_5796_gb300 as lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1309_5796_gb300 import build
    build.build()
    c = lbm.Context(0)
    yield c
    c.close()


def _products(ctx, mesh, batch, prec, seed):
    nb = ctx.mesh_info(mesh)["nb"]
    B = ctx.bem_rows(mesh, 0, nb)
    ctx.instance_create(mesh, 2, lbm.LBM_FP64).destroy()   # the mesh has the low words of B from here on
    x = np.random.default_rng(seed).normal(size=(nb, batch)) * 10.0 ** np.linspace(-6, 6, batch)
    y, yt = ctx.bem_apply(mesh, x, prec)
    # FP64: the sums to a few eps of sum |B| |x| (double-FP32 words: 2^-46 and less);
    # FP32: B and x rounded, compensated or short plain sums: (2 + 10) 2^-24
    tol = 4e-14 if prec == lbm.LBM_FP64 else 12 * 2.0 ** -24
    assert np.all(np.abs(y - B @ x) <= tol * (np.abs(B) @ np.abs(x)) + 1e-300)
    assert np.all(np.abs(yt - B.T @ x) <= tol * (np.abs(B).T @ np.abs(x)) + 1e-300)


# 8 to 2402 surface nodes: below and above a tile of 128 rows, a chunk of 256 columns;
# batches at the edges of the 8-, 16- and 32-wide tiles and of several tiles
@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_MIXED])
@pytest.mark.parametrize("n,batch", [(1, 1), (2, 1), (4, 1), (5, 1), (9, 1), (20, 1), (1, 2), (2, 8), (4, 9), (5, 16), (6, 17),
                                     (5, 32), (9, 33), (4, 48), (3, 65), (20, 6), (2, 256)])
def test_dense_products(ctx, n, batch, prec):
    mesh = ctx.mesh_cube(2e-9, n)
    _products(ctx, mesh, batch, prec, 100 * n + batch)
    ctx.mesh_destroy(mesh)


@pytest.mark.parametrize("batch", [1, 5])
def test_zero_and_special_columns(ctx, batch):
    """Zero vectors give zeros, and a NaN in one instance stays in it."""
    mesh = ctx.mesh_cube(2e-9, 5)
    nb = ctx.mesh_info(mesh)["nb"]
    x = np.zeros((nb, batch))
    for prec in (lbm.LBM_FP64, lbm.LBM_MIXED):
        y, yt = ctx.bem_apply(mesh, x, prec)
        assert not y.any() and not yt.any()
    x[7, 0] = np.nan
    y, yt = ctx.bem_apply(mesh, x, lbm.LBM_FP64)
    assert np.isnan(y[:, 0]).any() and np.isnan(yt[:, 0]).any()
    assert not np.isnan(y[:, 1:]).any() and not np.isnan(yt[:, 1:]).any()
    ctx.mesh_destroy(mesh)


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_MIXED])
@pytest.mark.parametrize("nodes,batch", [(5, 1), (7, 3), (305, 1), (305, 4)])
def test_odd_surfaces(ctx, nodes, batch, prec):
    """A chain of tetrahedra (a Boerdijk-Coxeter helix) has any number of surface nodes."""
    k = np.arange(nodes)
    th, r, h = np.arccos(-2 / 3), 3 * np.sqrt(3) / 10, 1 / np.sqrt(10)
    xyz = 2e-9 * np.stack([r * np.cos(k * th), r * np.sin(k * th), k * h], 1)
    mesh = ctx.mesh_upload(xyz, np.stack([k[:-3], k[1:-2], k[2:-1], k[3:]], 1))
    assert ctx.mesh_info(mesh)["nb"] == nodes
    _products(ctx, mesh, batch, prec, nodes + batch)
    ctx.mesh_destroy(mesh)
