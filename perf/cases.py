"""The work that programs give this library, as cases for timing and comparison.

A case is one call (or the few calls that belong together) through the Python
binding: a field evaluation, the energies of a batch, an evaluation that
allocates nothing, a batch of minimisations, a hysteresis branch.  The meshes
are Kuhn cubes and a mapped ball, with the three open boundaries (dense and
hierarchical boundary matrix, space transformation), in the three precisions.

FP64 results are returned as they come.  The mixed precisions fix a field or a
potential to FP32 accuracy, and a minimisation fixes m to its torque tolerance;
these results are returned in FP32, as a program keeps them.

All contexts work on one stream of the program (evaluations that allocate
nothing share one device array and must not overlap).
"""
import math

import numpy as np
import torch

import paper_1309_5796_gb300 as lbm

JS, A_EX, K1, CELL = 1.61, 7.7e-12, 4.3e6, 2e-9   # Nd2Fe14B, 2 nm cells
MU0 = 4e-7 * math.pi
PRECISIONS = {"fp64": lbm.LBM_FP64, "mixed": lbm.LBM_MIXED, "mixed_tc": lbm.LBM_MIXED_TC}
_stream = None


def _case(call, n, batch, precision, mesh="cube", boundary="dense", name=None, **more):
    c = dict(call=call, mesh=mesh, n=n, batch=batch, precision=precision, boundary=boundary, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the field of one small particle in FP64, the smallest call of an interactive program
        _case("evaluate", 10, 1, "fp64", name="evaluate_fp64_n10"),
        # the same for a host application that must not allocate while it runs (device pointers)
        _case("noalloc", 17, 1, "fp64", name="noalloc_fp64_n17"),
        # one 40 nm grain in mixed precision: the field inside a user's own loop
        _case("evaluate", 20, 1, "mixed", name="evaluate_mixed_n20"),
        # a few grains in FP64 on an odd lattice, the reference values of a study
        _case("evaluate", 25, 6, "fp64", name="evaluate_fp64_n25_b6"),
        # the energies of 64 states of a 60 nm cube (the benchmark's batch)
        _case("energy", 30, 64, "mixed_tc", name="energy_tc_n30_b64"),
        # one large cube: 531 441 nodes, a 38 402^2 boundary matrix
        _case("evaluate", 80, 1, "mixed", name="evaluate_mixed_n80"),
        # the same kind of problem with the boundary matrix in hierarchical form
        _case("evaluate", 40, 1, "mixed", boundary="hmatrix", name="evaluate_hmatrix_n40"),
        # the open boundary of the paper's own solver, a batch of grains
        _case("energy", 30, 32, "mixed", boundary="shell", air=4, shell=8, name="energy_shell_n30_b32"),
        # the paper's sphere grain, an uploaded mesh of its size and resolution
        _case("evaluate", 26, 1, "mixed", mesh="ball", name="evaluate_ball26_mixed"),
        # a batch on a smaller uploaded mesh in FP64
        _case("evaluate", 14, 16, "fp64", mesh="ball", name="evaluate_ball14_fp64_b16"),
        # whole minimisations of a batch: relaxations and reversals side by side
        _case("minimise", 30, 32, "mixed_tc", name="minimise_tc_n30_b32"),
        # a short hysteresis branch of a 20 nm cube in FP64, each point to a tight torque
        _case("hysteresis", 10, 1, "fp64", points=3, name="hysteresis_fp64_n10"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    """One more case: a call, a mesh size over the range it is used for, and a batch that keeps
    it below the largest listed one."""
    call = rng.choice(["evaluate", "evaluate", "energy", "noalloc", "hmatrix", "shell", "ball", "minimise", "hysteresis"])
    if call == "noalloc":
        return _case("noalloc", rng.randint(5, 24), 1, "fp64")
    if call == "hysteresis":
        return _case("hysteresis", rng.randint(5, 12), rng.choice([1, 1, 2]), "fp64", points=rng.randint(2, 3))
    if call == "minimise":
        n = rng.randint(8, 22)
        return _case("minimise", n, _log_int(rng, 1, 32), rng.choice(["mixed", "mixed_tc"]))
    if call == "hmatrix":
        n = rng.randint(12, 44)
        return _case("evaluate", n, _log_int(rng, 1, 4), rng.choice(["fp64", "mixed"]), boundary="hmatrix")
    if call == "shell":
        n = rng.randint(8, 28)
        return _case(rng.choice(["evaluate", "energy"]), n, _log_int(rng, 1, 32), rng.choice(["fp64", "mixed"]),
                     boundary="shell", air=rng.randint(2, 4), shell=rng.randint(4, 8))
    if call == "ball":
        n = 2 * rng.randint(4, 14)
        return _case("evaluate", n, _log_int(rng, 1, 24), rng.choice(["fp64", "mixed", "mixed_tc"]), mesh="ball")
    n = _log_int(rng, 5, 72)
    most = max(1, min(64, int(1.9e6 / (n + 1) ** 3)))
    precision = rng.choice(["fp64", "mixed", "mixed_tc"])
    return _case(call, n, _log_int(rng, 1, most if precision != "fp64" else max(1, most // 4)), precision)


# ---- inputs --------------------------------------------------------------------------
def _kuhn(n):
    """Lattice nodes (N, 3) and the six path tetrahedra of every cell, node (i, j, k) at
    i + (n+1)(j + (n+1)k)."""
    g = np.arange(n + 1)
    k, j, i = np.meshgrid(g, g, g, indexing="ij")
    nodes = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1).astype(np.float64)
    c = np.arange(n)
    ck, cj, ci = np.meshgrid(c, c, c, indexing="ij")
    base = np.stack([ci.ravel(), cj.ravel(), ck.ravel()], axis=1)
    step = np.array([1, n + 1, (n + 1) ** 2])
    tets = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        v0 = base @ step
        v1 = v0 + step[p[0]]
        v2 = v1 + step[p[1]]
        tets.append(np.stack([v0, v1, v2, v2 + step[p[2]]], axis=1))
    return nodes, np.stack(tets, axis=1).reshape(-1, 4)


def _ball(n):
    """A ball of n cells of 0.77 nm across: the lattice of [-1, 1]^3 moved nine tenths of the
    way onto the ball (rounded edges and corners, no flat tetrahedra)."""
    nodes, tets = _kuhn(n)
    p = nodes * (2.0 / n) - 1.0
    x, y, z = (p * p).T
    q = p * np.sqrt(np.stack([1 - y / 2 - z / 2 + y * z / 3, 1 - z / 2 - x / 2 + z * x / 3, 1 - x / 2 - y / 2 + x * y / 3], 1))
    return (0.1 * p + 0.9 * q) * (0.5 * n * 0.77e-9), tets.astype(np.int32)


def _points(case):
    """Node coordinates in units of the body's edge or diameter, in [0, 1]."""
    if case["mesh"] == "ball":
        xyz, _ = _ball(case["n"])
        return torch.from_numpy(xyz / (case["n"] * 0.77e-9) + 0.5)
    return torch.from_numpy(_kuhn_nodes(case["n"]) / case["n"])


def _kuhn_nodes(n):
    g = np.arange(n + 1, dtype=np.float64)
    k, j, i = np.meshgrid(g, g, g, indexing="ij")
    return np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1)


def _inputs(case, seed, dev="cuda"):
    """m (B, N, 3) on the GPU, easy axes (B, 3) within 5 degrees of z, fields (B, 3) in tesla."""
    g = torch.Generator(device=dev).manual_seed(seed)
    B, x = case["batch"], _points(case).to(dev)
    noise = torch.randn((B, x.shape[0], 3), generator=g, device=dev, dtype=torch.float64)
    u = torch.rand((B, 8), generator=g, device=dev, dtype=torch.float64)
    if case["call"] in ("minimise", "hysteresis"):
        m = 0.01 * noise   # +z, slightly disturbed
        m[..., 2] += 1.0
    else:
        # a state on the way of a minimisation: the moments turn smoothly through the body
        t = (x @ (3.0 * u[:, :3] - 1.5).T).T + 0.5 * u[:, 3:4]
        f = 2 * math.pi * u[:, 4:5] + (x @ (u[:, 5:8] - 0.5).T).T
        m = torch.stack([torch.sin(t) * torch.cos(f), torch.sin(t) * torch.sin(f), torch.cos(t)], -1) + 0.01 * noise
    m = m / m.norm(dim=-1, keepdim=True)
    tilt, turn = math.radians(5) * u[:, 3], 2 * math.pi * u[:, 4]
    axes = torch.stack([torch.sin(tilt) * torch.cos(turn), torch.sin(tilt) * torch.sin(turn), torch.cos(tilt)], -1)
    # along z: relaxations in [-3, 0] T, every other one a reversal in [-8, -7.5] T (in between,
    # near the switching field, rounding alone decides where a run ends)
    h = torch.zeros((B, 3), device=dev, dtype=torch.float64)
    h[:, 2] = -3.0 * u[:, 5]
    h[1::2, 2] = -7.5 - 0.5 * u[1::2, 5]
    return m.contiguous(), axes.cpu().numpy(), h.cpu().numpy()


def prepare(case, seed):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    m, axes, h = _inputs(case, seed)
    s = dict(case=case, m=m, axes=axes, h=h)
    torch.cuda.synchronize()
    ctx = lbm.Context(0, _stream.cuda_stream)
    s["ctx"] = ctx
    if case["mesh"] == "ball":
        mesh = ctx.mesh_upload(*_ball(case["n"]))
    else:
        mesh = ctx.mesh_cube(CELL, case["n"])
    if case["boundary"] == "hmatrix":
        ctx.mesh_hmatrix(mesh, 1e-6)
    if case["boundary"] == "shell":
        ctx.mesh_shell(mesh, case["air"], case["shell"])
    s["mesh"] = mesh
    precision = PRECISIONS[case["precision"]]
    if case["call"] == "noalloc":
        N = m.shape[1]
        s["h_out"] = torch.empty((N, 3), device="cuda", dtype=torch.float64)
        s["u_out"] = torch.empty((2, N), device="cuda", dtype=torch.float64)
        s["e_out"] = torch.empty(5, device="cuda", dtype=torch.float64)
        return s
    inst = ctx.instance_create(mesh, case["batch"], precision)
    inst.set_material(JS, A_EX, K1, axes)
    inst.set_field(h)
    s["inst"] = inst
    s["opts"] = lbm.default_opts(precision, tol=1e-10) if case["call"] == "hysteresis" else lbm.default_opts(precision)
    return s


def run(state):
    case, call = state["case"], state["case"]["call"]
    if call == "noalloc":
        state["ctx"].evaluate_noalloc(state["mesh"], JS, A_EX, K1, state["axes"][0], state["h"][0], state["m"].data_ptr(),
                                      state["h_out"].data_ptr(), state["u_out"].data_ptr(), state["e_out"].data_ptr())
        return {"energy": state["e_out"], "field": state["h_out"], "potential": state["u_out"]}
    inst = state["inst"]
    real = np.float64 if case["precision"] == "fp64" else np.float32
    inst.set_m_device(state["m"].data_ptr())
    if call == "energy":
        return {"energy": inst.energy().astype(real, copy=False)}
    if call == "evaluate":
        res, h, u = inst.evaluate(state["opts"])
        return {"energy": np.array([r["energy"] for r in res], real), "torque": np.array([r["torque"] for r in res], real),
                "field": h.astype(real, copy=False), "potential": u.astype(real, copy=False)}
    if call == "minimise":
        res = inst.minimise(state["opts"])
        return {"energy": np.array([r["energy"][4] for r in res]), "m": inst.get_m().astype(np.float32)}
    fields = np.linspace(1.0, -1.0, case["points"])
    m_par, energy, _ = inst.hysteresis([0.0, 0.0, 1.0], fields, state["opts"])
    return {"m_par": m_par, "energy": energy, "m": inst.get_m()}


def work(case):
    """Bytes and operations one pass cannot do without: m, the fields and potentials once, the
    boundary matrix once per evaluation, its two products, and each potential's system once
    (two forward, two adjoint; one on the grid of the space transformation)."""
    n, B = case["n"], case["batch"]
    N, nb = (n + 1) ** 3, 6 * n * n + 2
    word = 8 if case["precision"] == "fp64" else 4
    if case["boundary"] == "shell":
        rows = (n + 2 * (case["air"] + case["shell"]) + 1) ** 3
        matrix, solves = 0, 30.0 * rows * B
    else:
        part = 0.1 if case["boundary"] == "hmatrix" else 1.0
        matrix, solves = part * nb * nb, 4 * 15.0 * N * B
    flops = 4.0 * matrix * B + solves + 300.0 * N * B
    size = word * matrix + 24.0 * N * B
    if case["call"] in ("minimise", "hysteresis"):
        # at least some thirty steps from the disturbed state; m is read and written once
        steps = 30 * case.get("points", 1)
        return {"bytes": steps * word * matrix + 48.0 * N * B, "flops": steps * flops}
    if case["call"] == "energy":
        return {"bytes": size + 40.0 * B, "flops": flops}
    return {"bytes": size + 40.0 * N * B, "flops": flops}


# ---- the same evaluation in 64 bits, from the formulas ---------------------------------
def _cg(K, d, f, neumann):
    """Columns of K x = f by Jacobi-preconditioned CG to 1e-15 (neumann: modulo constants)."""
    x, r = torch.zeros_like(f), f.clone()
    stop = 1e-30 * (f * f).sum(0)
    p, rho = torch.zeros_like(f), torch.ones_like(stop)
    for it in range(20000):
        if neumann:
            r -= r.mean(0)
        z = r / d[:, None]
        new = (r * z).sum(0)
        rr = (r * r).sum(0)
        if it % 8 == 0 and bool((rr <= stop).all()):
            break
        live = rr > stop * 1e-2
        p = z + torch.where(live, new / rho, 0.0 * rho) * p if it else z
        rho = torch.where(live, new, torch.ones_like(new))
        q = K @ p
        alpha = torch.where(live, new / (p * q).sum(0), 0.0 * new)
        x += alpha * p
        r -= alpha * q
    return x


def _sparse(i, j, v, n):
    return torch.sparse_coo_tensor(torch.stack([i, j]), v, (n, n)).coalesce().to_sparse_csr()


def _double_layer(X, F, bnd):
    """B[i, j]: 1/(4 pi) times the integral of (x_i - y).n / |x_i - y|^3 phi_j(y) over the surface.
    Over one plane triangle it is -phi(p) Omega + h grad(phi) . sum_e nu_e P_e, with p the foot
    point of x_i in its plane, h the height, Omega the solid angle, nu_e the outward normals of
    the edges in the plane and P_e the integral of 1/r along them."""
    nb = bnd.numel()
    place = torch.zeros(X.shape[0], dtype=torch.long, device=X.device)
    place[bnd] = torch.arange(nb, device=X.device)
    Y = X[F]
    cr = torch.linalg.cross(Y[:, 1] - Y[:, 0], Y[:, 2] - Y[:, 0])
    a2 = cr.norm(dim=-1, keepdim=True)
    nrm = cr / a2
    E = Y.roll(-1, 1) - Y                          # edge k: vertex k to vertex k + 1
    s = E.norm(dim=-1)
    nu = torch.linalg.cross(E, nrm[:, None].expand_as(E)) / s[..., None]
    # gradient of hat k: from the edge opposite to vertex k
    gk = torch.linalg.cross(nrm[:, None].expand_as(E), E.roll(-1, 1)) / a2[:, None]
    out = torch.zeros((nb, nb), device=X.device, dtype=torch.float64)
    step = max(1, int(4e6) // F.shape[0])
    for i0 in range(0, nb, step):
        ids = bnd[i0:i0 + step]
        R = Y[None] - X[ids][:, None, None]        # (rows, triangles, vertices, 3)
        r = R.norm(dim=-1)
        h = (R[:, :, 0] * nrm).sum(-1)
        own = (F[None] == ids[:, None, None]).any(-1) | (h == 0)
        num = (R[:, :, 0] * torch.linalg.cross(R[:, :, 1], R[:, :, 2])).sum(-1)
        den = r.prod(-1)
        for k in range(3):
            den = den + r[:, :, k] * (R[:, :, (k + 1) % 3] * R[:, :, (k + 2) % 3]).sum(-1)
        omega = 2 * torch.atan2(num, den)
        P = torch.log1p(2 * s / (r + r.roll(-1, 2) - s).clamp_min(1e-300))
        edge = torch.einsum("itk,tkd->itd", P, nu)
        foot = h[..., None] * nrm - R[:, :, 0]     # relative to vertex 0
        phi = torch.einsum("itd,tkd->itk", foot, gk)
        phi[..., 0] += 1.0
        val = -phi * omega[..., None] + h[..., None] * torch.einsum("itd,tkd->itk", edge, gk)
        val = torch.where(own[..., None], torch.zeros_like(val), val) / (4 * math.pi)
        out[i0:i0 + step].index_add_(1, place[F].reshape(-1), val.reshape(ids.numel(), -1))
    return out


def exact(case, seed):
    if case["call"] in ("minimise", "hysteresis") or (case["n"] + 1) ** 3 > 80000:
        return None
    m, axes, h_ext = _inputs(case, seed)
    dev = m.device
    B, n = case["batch"], case["n"]
    if case["mesh"] == "ball":
        xyz, tets = _ball(n)
        unit = 0.77e-9
    else:
        xyz, tets = _kuhn(n)
        unit = CELL
        xyz = xyz * unit
    X, T = torch.from_numpy(xyz / unit).to(dev), torch.from_numpy(tets.astype(np.int64)).to(dev)
    N = X.shape[0]

    def elements(X, T):
        P = X[T]
        D = P[:, 1:] - P[:, :1]
        det = torch.linalg.det(D)
        g = torch.linalg.inv(D).transpose(1, 2)     # rows: gradients of hats 1, 2, 3
        return torch.cat([-g.sum(1, keepdim=True), g], 1), det.abs() / 6

    grad, vol = elements(X, T)
    ii, jj = T[:, :, None].expand(-1, 4, 4).reshape(-1), T[:, None, :].expand(-1, 4, 4).reshape(-1)
    K = _sparse(ii, jj, (torch.einsum("tad,tbd->tab", grad, grad) * vol[:, None, None]).reshape(-1), N)
    V = torch.zeros(N, device=dev, dtype=torch.float64).index_add_(0, T.reshape(-1), (vol / 4)[:, None].expand(-1, 4).reshape(-1))
    G = [_sparse(ii, jj, (grad[:, :, d:d + 1] * (vol / 4)[:, None, None]).expand(-1, 4, 4).reshape(-1), N) for d in range(3)]
    GT = [_sparse(jj, ii, (grad[:, :, d:d + 1] * (vol / 4)[:, None, None]).expand(-1, 4, 4).reshape(-1), N) for d in range(3)]
    M = m.permute(2, 1, 0)                          # (3, N, B)
    b = sum(G[d] @ M[d] for d in range(3))
    if case["boundary"] == "shell":
        u1 = _shell_potential(case, b, dev, elements)
        u2, uT = torch.zeros_like(u1), u1
    else:
        u1, u2, uT = _fem_bem(X, T, K, ii, jj, grad, vol, V, b, dev)
    hd = -torch.stack([GT[d] @ (0.5 * (u1 + u2 + uT)) for d in range(3)]) / V[:, None]
    ax = torch.from_numpy(axes).to(dev).T[:, None]  # (3, 1, B)
    hx = torch.from_numpy(h_ext).to(dev).T[:, None]
    kd = JS * JS / (2 * MU0)
    ma = (M * ax).sum(0)
    KM = torch.stack([K @ M[d] for d in range(3)])
    h = JS * hd + hx + (2 * K1 / JS * MU0) * ma * ax - (2 * A_EX * MU0 / JS / unit ** 2) * KM / V[:, None]
    e_ex = A_EX * unit * (M * KM).sum((0, 1))
    e_an = K1 * unit ** 3 * (V[:, None] * torch.linalg.cross(M, ax.expand_as(M), dim=0).square().sum(0)).sum(0)
    e_z = -JS / MU0 * unit ** 3 * (V[:, None] * (M * hx).sum(0)).sum(0)
    e_d = -kd * unit ** 3 * (V[:, None] * (M * hd).sum(0)).sum(0)
    energy = torch.stack([e_ex, e_an, e_z, e_d, e_ex + e_an + e_z + e_d], 1).cpu()
    if case["call"] == "energy":
        return {"energy": energy}
    field = h.permute(2, 1, 0).contiguous().cpu()
    torque = torch.linalg.cross(M, h, dim=0).norm(dim=0).amax(0) / JS
    pot = torch.stack([u1, u2], 0).permute(2, 0, 1) * unit
    if case["call"] == "noalloc":
        return {"energy": energy[0], "field": field[0], "potential": pot[0].contiguous().cpu()}
    return {"energy": energy, "torque": torque.cpu(), "field": field, "potential": pot.contiguous().cpu()}


def _fem_bem(X, T, K, ii, jj, grad, vol, V, b, dev):
    """u1, u2 and the adjoint chain's uT (columns: instances)."""
    N = X.shape[0]
    # outward faces of the surface: those of one tetrahedron only
    faces, inner = [], []
    for a, c, e, o in ((1, 2, 3, 0), (0, 3, 2, 1), (0, 1, 3, 2), (0, 2, 1, 3)):
        faces.append(T[:, [a, c, e]])
        inner.append(T[:, o])
    F, O = torch.cat(faces), torch.cat(inner)
    S = F.sort(1).values
    key = (S[:, 0] * N + S[:, 1]) * N + S[:, 2]
    _, inv, cnt = torch.unique(key, return_inverse=True, return_counts=True)
    F, O = F[cnt[inv] == 1], O[cnt[inv] == 1]
    nrm = torch.linalg.cross(X[F[:, 1]] - X[F[:, 0]], X[F[:, 2]] - X[F[:, 0]])
    flip = (nrm * (X[O] - X[F[:, 0]])).sum(-1) > 0
    F = torch.where(flip[:, None], F[:, [0, 2, 1]], F)
    bnd = torch.unique(F)
    # solid angle of the body at every surface node: the sum over its tetrahedra
    angle = torch.zeros(N, device=dev, dtype=torch.float64)
    P = X[T]
    for k in range(4):
        e = [P[:, (k + s) % 4] - P[:, k] for s in (1, 2, 3)]
        r = [v.norm(dim=-1) for v in e]
        num = (e[0] * torch.linalg.cross(e[1], e[2])).sum(-1).abs()
        den = r[0] * r[1] * r[2] + sum((e[a] * e[c]).sum(-1) * r[3 - a - c] for a, c in ((0, 1), (0, 2), (1, 2)))
        angle.index_add_(0, T[:, k], 2 * torch.atan2(num, den))
    Bm = _double_layer(X, F, bnd)
    Bm.diagonal().add_(angle[bnd] / (4 * math.pi) - 1.0)
    surf = torch.zeros(N, dtype=torch.bool, device=dev)
    surf[bnd] = True
    val = (torch.einsum("tad,tbd->tab", grad, grad) * vol[:, None, None]).reshape(-1)
    both = ~surf[ii] & ~surf[jj]
    KI = _sparse(ii[both], jj[both], val[both], N)
    diag = torch.zeros(N, device=dev, dtype=torch.float64).index_add_(0, ii[ii == jj], val[ii == jj])
    free = (~surf).double()[:, None]
    u1 = _cg(K, diag, b - b.mean(0), True)
    u1 = u1 - (V[:, None] * u1).sum(0) / V.sum()
    g = torch.zeros_like(b)
    g[bnd] = Bm @ u1[bnd]
    u2 = g + _cg(KI, diag, -free * (K @ g), False)
    w = _cg(KI, diag, free * b, False)
    t = (b - K @ w)[bnd]
    c = b.clone()
    c[bnd] += Bm.T @ t
    uT = _cg(K, diag, c - c.mean(0), True)
    return u1, u2, uT - (V[:, None] * uT).sum(0) / V.sum()


def _shell_potential(case, b, dev, elements):
    """u on the magnet's nodes from the one solve on the grid over magnet, air and mapped shell."""
    n, a, s = case["n"], case["air"], case["shell"]
    nt = n + 2 * (a + s)
    nodes, tets = _kuhn(nt)
    X, T = torch.from_numpy(nodes).to(dev), torch.from_numpy(tets.astype(np.int64)).to(dev)
    grad, vol = elements(X, T)
    R1, R2 = n / 2 + a, n / 2 + a + s
    x = X[T].mean(1) - nt / 2
    rho, d = x.abs().max(1)                          # the first largest coordinate is the sector's
    outer = rho > R1
    g = R1 * (R2 - R1) / (R2 - rho)
    sig, dsig = g / rho, (g / (R2 - rho) - g / rho) / rho
    drho = torch.zeros_like(x)
    drho[torch.arange(x.shape[0], device=dev), d] = torch.sign(x[torch.arange(x.shape[0], device=dev), d])
    eye = torch.eye(3, device=dev, dtype=torch.float64).expand(x.shape[0], 3, 3)
    J = torch.where(outer[:, None, None], sig[:, None, None] * eye + dsig[:, None, None] * x[:, :, None] * drho[:, None, :], eye)
    Ji = torch.linalg.inv(J)
    Mt = torch.linalg.det(J).abs()[:, None, None] * Ji @ Ji.transpose(1, 2)
    val = (torch.einsum("tad,tde,tbe->tab", grad, Mt, grad) * vol[:, None, None]).reshape(-1)
    ii, jj = T[:, :, None].expand(-1, 4, 4).reshape(-1), T[:, None, :].expand(-1, 4, 4).reshape(-1)
    on = ((X - nt / 2).abs().max(1).values > R2 - 0.5)
    keep = ~on[ii] & ~on[jj]
    NG = X.shape[0]
    K = _sparse(ii[keep], jj[keep], val[keep], NG)
    diag = torch.ones(NG, device=dev, dtype=torch.float64)
    own = keep & (ii == jj)
    diag[~on] = 0.0
    diag.index_add_(0, ii[own], val[own])
    inner = torch.from_numpy(_kuhn_nodes(n)).to(dev).long() + (a + s)
    at = inner[:, 0] + (nt + 1) * (inner[:, 1] + (nt + 1) * inner[:, 2])
    f = torch.zeros((NG, b.shape[1]), device=dev, dtype=torch.float64)
    f[at] = b
    return _cg(K, diag, f, False)[at]
