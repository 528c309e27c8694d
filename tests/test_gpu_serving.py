"""Continuous-batching server (config 5 workload pattern) on the GPU.

A request gives the same result alone and in a mix of concurrent requests of
other cube sizes (each instance's arithmetic and reduction order is independent
of what else is in its batch), and the same result as the batch API.
"""

import numpy as np
import pytest

import paper_1309_5796_gb300 as lbm
from synth.inputs import A_JM, JS_T, K1_JM3, m_perturbed, tilted_axis

pytestmark = pytest.mark.gpu


def _req(n, seed, hz, tilt):
    N = (n + 1) ** 3
    return dict(n=n, cell_m=2e-9, Js=JS_T, A=A_JM, K1=K1_JM3, axis=tilted_axis(tilt, 0.3 * seed),
                h=np.array([0.0, 0.0, hz]), m0=m_perturbed(N, seed))


@pytest.fixture(scope="module")
def ctx():
    from paper_1309_5796_gb300 import build
    build.build()
    c = lbm.Context(0)
    yield c
    c.close()


def test_alone_and_in_the_mix(ctx):
    target = _req(8, 11, -5.0, 3.0)
    others = [_req(n, 20 + k, -8.0 + 1.3 * k, 1.0 + k) for k, n in enumerate((4, 6, 8, 8, 10, 5, 7))]
    N = (target["n"] + 1) ** 3
    ctx.serve_start(slots=4, chunk=4)
    try:
        t0 = ctx.submit(**target)
        alone, m_alone = ctx.wait(t0, N, timeout_s=300)
        tickets = [ctx.submit(**r) for r in others[:3]]
        t1 = ctx.submit(**target)
        tickets += [ctx.submit(**r) for r in others[3:]]
        mix, m_mix = ctx.wait(t1, N, timeout_s=300)
        rest = [ctx.wait(t, None, timeout_s=300)[0] for t in tickets]
        stats = ctx.serve_stats()
    finally:
        ctx.serve_stop()
    assert alone["status"] == lbm.LBM_OK and alone["torque"] < 1e-6
    assert all(r["status"] == lbm.LBM_OK and r["torque"] < 1e-6 for r in rest)
    # same arithmetic alone and in the mix
    assert mix["energy"][4] == alone["energy"][4]
    assert np.array_equal(m_mix, m_alone)
    assert stats["completed"] == 2 + len(others) and stats["pending"] == 0
    assert stats["groups"] >= 4
    # the batch API on the same problem (one instance): same minimum
    mesh = ctx.mesh_cube(2e-9, target["n"])
    inst = ctx.instance_create(mesh, 1, lbm.LBM_MIXED)
    inst.set_material(JS_T, A_JM, K1_JM3, target["axis"])
    inst.set_field(target["h"])
    inst.set_m(target["m0"])
    r = inst.minimise(lbm.default_opts(lbm.LBM_MIXED))[0]
    inst.destroy()
    ctx.mesh_destroy(mesh)
    assert r["status"] == lbm.LBM_OK
    scale = max(abs(r["energy"][4]), 1.0e-20)
    assert abs(r["energy"][4] - alone["energy"][4]) / scale < 1e-6


def test_fp64_requests_and_latency(ctx):
    reqs = [_req(n, 40 + n, -6.0, 2.0) for n in (3, 5, 6)]
    ctx.serve_start(slots=2, chunk=8)
    try:
        ts = [ctx.submit(**r, precision=lbm.LBM_FP64) for r in reqs]
        res = [ctx.wait(t, None, timeout_s=300)[0] for t in ts]
        pending = ctx.poll(ctx.submit(**reqs[0]))
    finally:
        ctx.serve_stop()
    assert all(r["status"] == lbm.LBM_OK and r["torque"] < 1e-6 for r in res)
    assert all(r["wall_ms"] > 0 for r in res)
    assert pending is None or pending[0]["status"] == lbm.LBM_OK


def test_size_groups_overlap_on_the_device(ctx):
    """Requests of three cube sizes served together: the serving loop's device
    trace (CUDA events on each size group's stream) has chunks of different
    groups whose intervals intersect, i.e. their kernels ran concurrently."""
    from synth.inputs import m_perturbed, tilted_axis
    ctx.serve_start(slots=16, chunk=8)
    try:
        tickets = []
        for k, n in enumerate((10, 14, 18) * 3):
            N = (n + 1) ** 3
            tickets.append(ctx.submit(n, 2e-9, JS_T, A_JM, K1_JM3, tilted_axis(2.0 + k, 0.3 * k),
                                      np.array([0.0, 0.0, -1.0 - 0.4 * k]), m_perturbed(N, 4000 + k)))
        res = [ctx.wait(t, None, timeout_s=600)[0] for t in tickets]
        tr = ctx.serve_trace()
    finally:
        ctx.serve_stop()
    assert all(r["status"] == lbm.LBM_OK for r in res)
    sizes = sorted(set(tr[:, 0].astype(int)))
    assert len(sizes) == 3
    overlaps = 0
    for i in range(len(tr)):
        for j in range(i + 1, len(tr)):
            if tr[i, 0] != tr[j, 0] and max(tr[i, 1], tr[j, 1]) < min(tr[i, 2], tr[j, 2]):
                overlaps += 1
    assert overlaps > 0


def test_the_block_cap_holds_for_cubes(ctx):
    """max_pcg_blocks caps the blocks of a group's potential solves: with one block a solve
    takes a launch for each of the batch's systems, with the device's it takes one; the
    results have the same bits."""
    req = _req(6, 17, -5.0, 3.0)
    N = (req["n"] + 1) ** 3
    out = []
    for cap in (1, 100000):
        ctx.serve_start(slots=4, chunk=4, max_pcg_blocks=cap)
        try:
            k0 = ctx.launch_count()
            r, m = ctx.wait(ctx.submit(**req), N, timeout_s=300)
        finally:
            ctx.serve_stop()   # the loop has ended: its counter is still
        out.append((r, m, ctx.launch_count() - k0))
    (ra, ma, la), (rb, mb, lb) = out
    assert ra["status"] == rb["status"] == lbm.LBM_OK
    assert ra["energy"] == rb["energy"] and np.array_equal(ma, mb)
    # an evaluation is at most 7 launches with one a solve; its two solves have two systems to serve
    assert la >= lb + 2 * ra["evaluations"]


def test_a_group_is_admitted_with_the_memory_it_takes(ctx):
    """The memory a size group is said to need covers what it takes: with 8 MB less than
    that free (the rest reserved) a request waits, with it and some more it runs."""
    import time

    import torch
    req = _req(30, 12, -4.0, 3.0)
    torch.cuda.mem_get_info()

    def free():
        return torch.cuda.mem_get_info()

    def serve(reserve):
        ctx.serve_start(slots=64, chunk=8, mem_reserve=reserve)
        try:
            t = ctx.submit(**req)
            time.sleep(1.0)
            st = ctx.serve_stats()
            if not st["active_slots"] and not st["completed"]:
                return st, None
            used = f0 - free()[0]
            ctx.wait(t, None, timeout_s=300)
            return st, used
        finally:
            ctx.serve_stop()

    f0, tot = free()
    serve(0.0)                       # modules, kernels and pools of a first run
    f0 = free()[0]
    st, used = serve(0.0)
    assert used > 0 and st["stalls"] == 0
    f0 = free()[0]
    st, none = serve((f0 - used + (8 << 20)) / tot)
    assert none is None and st["stalls"] > 0
    st, again = serve((f0 - used - (256 << 20)) / tot)
    assert again is not None and st["stalls"] == 0
