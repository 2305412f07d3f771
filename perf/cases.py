"""What a user of the library has it do, as cases that can be timed and compared.

Every case goes through the Python binding of the C-ABI as a solver or a serving loop calls it:

* ``assemble``: upload a state that lives on the GPU, one Newton-Schur tangent assembly, the
  assembled system as device tensors (hexahedra and tetrahedra, FP64 and mixed precision, steady
  and backward Euler, body force, batches of independent problems replayed from a graph);
* ``residual``: the FP64 residual vector and its norm (Newton's stopping test, line searches);
* ``linear``: one Newton step by hand: assembly, preconditioned GMRES, bubble recovery, update;
* ``newton``: a whole inexact Newton solve;
* ``mlp_grad`` / ``mlp_forward``: gradient of a training batch and inference of the warm-start
  network.

Sizes are those of the benchmark's and the tests' workloads, and odd ones between them.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0809_4802_gb300 import inputs, vms

DEV = "cuda:0"
PRECISIONS = {"fp64": vms.PREC_FP64, "mixed": vms.PREC_MIXED}


# ----------------------------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest assembly a user runs: the paper's cavity at Re 100 on 8^3 elements, all FP64
        {"name": "assemble_cavity8_fp64", "kind": "assemble", "mesh": "cavity", "nx": 8, "precision": "fp64",
         "re": 100.0, "jitter": 0.0, "dt": 0.0, "force": False, "quad": 3, "graph": False},
        # a ragged FP64 problem: odd edge counts, a hole, a time step and a body force
        {"name": "assemble_holedbox_fp64", "kind": "assemble", "mesh": "holed_box", "nx": 31, "ny": 23, "nz": 19,
         "precision": "fp64", "re": 250.0, "jitter": 0.2, "dt": 0.01, "force": True, "quad": 3, "graph": False},
        # the benchmark's mid-size problem: the jittered 32^3 cavity at Re 400, mixed precision
        {"name": "assemble_cavity32_mixed", "kind": "assemble", "mesh": "cavity", "nx": 32, "precision": "mixed",
         "re": 400.0, "jitter": 0.15, "dt": 0.0, "force": False, "quad": 3, "graph": False},
        # a serving mix: cavities of uneven size, each with its own viscosity, one graph replay
        {"name": "assemble_batch_mixed", "kind": "assemble", "mesh": "batch", "edges": "8,24,12,32,16,9,13,24,8,17",
         "precision": "mixed", "re": 100.0, "jitter": 0.15, "dt": 0.0, "force": False, "quad": 3, "graph": True},
        # the benchmark's default workload: one backward-Euler step of the channel past a cube
        {"name": "assemble_channel_mixed", "kind": "assemble", "mesh": "channel", "nx": 300, "ny": 56,
         "precision": "mixed", "re": 1000.0, "jitter": 0.0, "dt": 0.01, "force": False, "quad": 3, "graph": False},
        # the tetrahedral element on about the paper's mesh E
        {"name": "assemble_tet39_mixed", "kind": "assemble", "mesh": "tet_cavity", "nx": 39, "precision": "mixed",
         "re": 400.0, "jitter": 0.15, "dt": 0.0, "force": False, "quad": 3, "graph": False},
        # Newton's stopping test on a mid-size transient problem with a body force
        {"name": "residual_holedbox", "kind": "residual", "mesh": "holed_box", "nx": 47, "ny": 33, "nz": 29,
         "precision": "fp64", "re": 500.0, "jitter": 0.2, "dt": 0.01, "force": True, "quad": 3, "graph": False},
        # one Newton step of the 32^3 cavity in mixed precision: FP64 factorisation, FP32 sweeps and
        # Krylov vectors, FP64 refinement (a tolerance that late inexact Newton steps ask for)
        {"name": "linear_cavity32_mixed", "kind": "linear", "mesh": "cavity", "nx": 32, "precision": "mixed",
         "re": 400.0, "jitter": 0.15, "rtol": 1e-6, "restart": 150},
        # one Newton step on tetrahedra in mixed precision, solved tightly: several Krylov cycles
        {"name": "linear_tet21_mixed", "kind": "linear", "mesh": "tet_cavity", "nx": 21, "precision": "mixed",
         "re": 400.0, "jitter": 0.15, "rtol": 1e-10, "restart": 150},
        # a whole Newton solve to 1e-8 in plain FP64
        {"name": "newton_cavity24_fp64", "kind": "newton", "mesh": "cavity", "nx": 24, "precision": "fp64",
         "re": 200.0, "jitter": 0.15, "rtol": 1e-8},
        # a training minibatch of the warm-start network (gradient read back)
        {"name": "mlp_grad_1024", "kind": "mlp_grad", "rows": 1024},
        # the network on every node of the channel past a cube
        {"name": "mlp_forward_channel", "kind": "mlp_forward", "rows": 975583},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["assemble", "assemble", "assemble", "assemble", "residual", "linear", "linear", "newton",
                       "mlp_grad", "mlp_forward"])
    if kind.startswith("mlp"):
        return {"kind": kind, "rows": _log(rng, 200, 900000)}
    if kind in ("linear", "newton"):
        mesh = rng.choice(["cavity", "tet_cavity"])
        c = {"kind": kind, "mesh": mesh, "precision": rng.choice(["fp64", "mixed"]),
             "nx": rng.randint(6, 24) if mesh == "cavity" else rng.randint(5, 20),
             "re": float(_log(rng, 20, 200)), "jitter": rng.choice([0.05, 0.1, 0.15]),
             "rtol": 1e-8 if kind == "newton" else 1e-10}
        if mesh == "cavity" and c["precision"] == "mixed":
            # a tight FP32-matrix solve of a distorted hexahedral mesh may not converge (near-null
            # pressure modes): mixed precision there on larger meshes and to a looser tolerance
            if kind == "newton":
                c["precision"] = "fp64"
            else:
                c.update(nx=rng.randint(20, 34), jitter=0.15, rtol=1e-6)
        if kind == "linear":
            c["restart"] = 150
        return c
    c = {"kind": kind, "precision": rng.choice(["fp64", "mixed", "mixed"]) if kind == "assemble" else "fp64",
         "re": float(_log(rng, 50, 1000)), "jitter": rng.choice([0.0, 0.1, 0.2]), "dt": rng.choice([0.0, 0.01]),
         "force": rng.choice([False, True]), "quad": rng.choice([2, 3, 3, 3]), "graph": rng.choice([False, False, True])}
    c["mesh"] = rng.choice(["cavity", "holed_box", "tet_cavity", "batch", "channel"] if kind == "assemble"
                           else ["cavity", "holed_box", "tet_cavity", "channel"])
    if c["mesh"] == "cavity":
        c["nx"] = _log(rng, 5, 72)
    elif c["mesh"] == "tet_cavity":
        c["nx"] = _log(rng, 4, 40)
    elif c["mesh"] == "batch":
        c["edges"] = ",".join(str(rng.choice([6, 8, 9, 12, 13, 16, 17, 24])) for _ in range(rng.randint(2, 16)))
    elif c["mesh"] == "channel":
        c["nx"], c["ny"] = _log(rng, 60, 200), rng.randint(16, 40)
    else:
        c["nx"], c["ny"], c["nz"] = (_log(rng, 7, 60) for _ in range(3))
    return c


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _state(mesh, rng, kind):
    u = np.zeros((mesh.n_nodes, 4))
    if kind == "random":      # the cavity benchmark's state: every mode of the element excited
        u[:, :3] = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 3))
        u[:, 3] = rng.normal(0.0, 0.1, mesh.n_nodes)
    else:                     # near rest, as the 8^3 cavity starts
        inner = ~inputs.boundary_nodes(mesh)
        u[inner, :3] = rng.uniform(-0.05, 0.05, (int(inner.sum()), 3))
    return u


def _workload(case, seed):
    """(xyz, conn, bc, u, beta, u_prev, nu, nu_e, node_offsets, elem_offsets) on the host."""
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    nu, nu_e, offs = 1.0 / case["re"], None, (None, None)
    name, jit = case["mesh"], case["jitter"]
    if name == "batch":
        edges = [int(t) for t in case["edges"].split(",")]
        b = inputs.merge_workloads([
            inputs.cavity_workload(n, float(rng.uniform(100.0, 1000.0)), jitter_frac=jit, state="random",
                                   seed=1000 * seed + i) for i, n in enumerate(edges)])
        mesh, bc, u = b.work.mesh, b.work.bc, b.work.u
        nu_e, offs = b.nu_e, (b.node_offsets, b.elem_offsets)
    else:
        if name == "channel":
            wl = inputs.channel_workload(case["nx"], case["ny"])
            mesh, bc = wl.mesh, wl.bc
            inputs.jitter(mesh, jit, rng)
        elif name == "holed_box":
            d = (case["nx"], case["ny"], case["nz"])
            hole = tuple((n // 3, n // 3 + max(1, n // 5)) for n in d)
            mesh = inputs.box_mesh(*d, hi=(1.0, d[1] / d[0], d[2] / d[0]), jitter_frac=jit,
                                   seed=int(rng.integers(1 << 30)), hole=hole)
            bc = inputs.wall_bc(mesh, pin_pressure_node=0)
        else:
            hexm = inputs.cavity_mesh(case["nx"], jit, int(rng.integers(1 << 30)))
            bc = inputs.cavity_bc(hexm)
            mesh = hexm if name == "cavity" else inputs.tet_mesh_from_lattice(hexm)
        near_rest = case["kind"] in ("linear", "newton")
        src = hexm if name == "tet_cavity" else mesh
        u = inputs.impose(_state(src, rng, "noise" if near_rest else "random"), bc)
    beta = rng.uniform(-0.1, 0.1, (mesh.n_elems, 3)) if case["kind"] in ("assemble", "residual") else np.zeros((mesh.n_elems, 3))
    u_prev = u + rng.uniform(-0.01, 0.01, u.shape) if case.get("dt") else None
    return mesh.xyz, mesh.conn, bc, u, beta, u_prev, nu, nu_e, *offs


def _force(case):
    return (0.3, -0.2, 0.5) if case.get("force") else (0.0, 0.0, 0.0)


def _mlp_inputs(case, seed):
    params = inputs.mlp_init(seed)
    r = np.random.Generator(np.random.PCG64([seed, 78]))
    for at in (1536, 18048, 18688):   # the biases of a network that has been trained for a while
        n = 4 if at == 18688 else 128
        params[at:at + n] = r.normal(0.0, 0.1, n).astype(np.float32)
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["rows"]
    x = torch.randn((n, 12), generator=g, device=DEV, dtype=torch.float32)
    t = torch.randn((n, 4), generator=g, device=DEV, dtype=torch.float32)
    return params, x, t


def prepare(case, seed):
    if case["kind"].startswith("mlp"):
        params, x, t = _mlp_inputs(case, seed)
        mlp = vms.Mlp(0)
        mlp.set_stream(torch.cuda.current_stream().cuda_stream)
        mlp.set_params(params)
        return {"case": case, "mlp": mlp, "x": x, "t": t, "y": torch.empty((case["rows"], 4), device=DEV)}
    xyz, conn, bc, u, beta, u_prev, nu, nu_e, no, eo = _workload(case, seed)
    ctx = vms.Context(0, PRECISIONS[case["precision"]])
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    ctx.mesh_upload(xyz, conn, bc.dofs, bc.vals)
    ctx.set_params(nu, dt=case.get("dt", 0.0), f=_force(case), quad_order=case.get("quad", 3))
    if nu_e is not None:
        ctx.set_element_viscosity(nu_e)
        ctx.set_instances(no, eo)
    if case.get("graph"):
        ctx.set_graph(True)
    dev = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    s = {"case": case, "ctx": ctx, "u": dev(u), "beta": dev(beta), "u_prev": dev(u_prev)}
    if case["kind"] == "residual":
        s["R"] = torch.empty(4 * ctx.n_nodes + 3 * ctx.n_elems, dtype=torch.float64, device=DEV)
    return s


# ----------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mlp_forward":
        state["mlp"].forward(state["x"], state["y"])
        return {"y": state["y"]}
    if kind == "mlp_grad":
        loss, grad = state["mlp"].grad(state["x"], state["t"])
        return {"loss": loss, "grad": grad}
    ctx = state["ctx"]
    ctx.state_upload(state["u"], state["beta"], state["u_prev"])
    if kind == "assemble":
        _, _, values, rhs = ctx.csr_device(ctx.assemble())
        return {"values": values, "rhs": rhs}
    if kind == "residual":
        # the C entry, which takes a device buffer for the vector (the binding's own method brings
        # it to the host)
        norm = ctypes.c_double()
        if ctx.lib.vms_residual(ctx.h, ctypes.byref(norm), state["R"].data_ptr()) != vms.OK:
            raise RuntimeError(ctx.lib.vms_last_error(ctx.h).decode())
        return {"norm": norm.value, "R": state["R"]}
    if kind == "linear":
        ctx.assemble()
        ctx.solve(rtol=case["rtol"], maxit=3000, restart=case["restart"], update=True)
    else:
        ctx.newton_solve(rtol=case["rtol"], maxit=25)
    u, beta = ctx.state_download()
    return {"u": u, "beta": beta}


# ----------------------------------------------------------------------------------------------
# the least work of a pass
# ----------------------------------------------------------------------------------------------
def _sizes(case):
    """(elements, nodes, node pairs sharing an element) of a case's mesh, holes included."""
    def lattice(a, b, c):
        return a * b * c, (a + 1) * (b + 1) * (c + 1), (3 * a + 1) * (3 * b + 1) * (3 * c + 1)
    m = case["mesh"]
    if m == "batch":
        parts = [lattice(int(t), int(t), int(t)) for t in case["edges"].split(",")]
        return tuple(sum(p[k] for p in parts) for k in range(3))
    if m == "tet_cavity":
        n = case["nx"]
        e = 3 * n * (n + 1) ** 2 + 3 * n * n * (n + 1) + n ** 3   # edges of the Kuhn subdivision
        return 6 * n ** 3, (n + 1) ** 3, (n + 1) ** 3 + 2 * e
    if m == "cavity":
        return lattice(case["nx"], case["nx"], case["nx"])
    if m == "channel":
        hx, hy = 20.0 / case["nx"], 4.0 / case["ny"]
        box = (case["nx"], case["ny"], case["ny"])
        j = int(round(2.5 / hy)) - int(round(1.5 / hy))
        hole = (int(round(5.0 / hx)) - int(round(4.0 / hx)), j, j)
    else:
        box = (case["nx"], case["ny"], case["nz"])
        hole = tuple(max(1, n // 5) for n in box)
    whole = lattice(*box)
    inner = (hole[0] * hole[1] * hole[2], (hole[0] - 1) * (hole[1] - 1) * (hole[2] - 1),
             max(0, 3 * hole[0] - 2) * max(0, 3 * hole[1] - 2) * max(0, 3 * hole[2] - 2))
    return tuple(w - h for w, h in zip(whole, inner))


def work(case):
    if case["kind"].startswith("mlp"):
        n = case["rows"]
        if case["kind"] == "mlp_forward":
            return {"bytes": n * 64 + 4 * 18692, "flops": 2.0 * 18432 * n}
        return {"bytes": n * 64 + 8 * 18692, "flops": 6.0 * 18432 * n}
    elems, nodes, pairs = _sizes(case)
    npe = 4 if case["mesh"] == "tet_cavity" else 8
    state = nodes * (24 + 32 + (32 if case.get("dt") else 0)) + elems * (4 * npe + 24)
    q = case.get("quad", 3) ** 3 / 27.0
    # counts of a direct evaluation of the formulas at every quadrature point (hexahedra), or of the
    # reference moments (tetrahedra)
    f_res, f_tan = (24300.0 * q, 86400.0 * q + 7000.0) if npe == 8 else (1500.0, 4366.0)
    if case["kind"] == "residual":
        return {"bytes": state + nodes * 32 + elems * 24, "flops": f_res * elems}
    system = 16 * pairs * (8 if case["precision"] == "fp64" else 4) + nodes * 32
    if case["kind"] == "assemble":
        return {"bytes": state + system, "flops": (f_res + f_tan) * elems}
    # solves: one assembly, one pass over the matrix and the new state (the iterations depend on the data)
    return {"bytes": state + 2 * system + nodes * 32 + elems * 24, "flops": (f_res + f_tan) * elems + 32.0 * pairs}


# ----------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------------------------
def _hex_rule(n):
    x, w = np.polynomial.legendre.leggauss(n)
    z, y, t = np.meshgrid(x, x, x, indexing="ij")
    p = np.stack([t.ravel(), y.ravel(), z.ravel()], 1)
    c = inputs.HEX_CORNERS.astype(float)
    f = 1.0 + p[:, None, :] * c[None]
    N = f.prod(2) / 8.0
    dN = np.stack([c[None, :, d] * np.delete(f, d, 2).prod(2) / 8.0 for d in range(3)], 2)
    g = 1.0 - p * p
    db = np.stack([-2.0 * p[:, d] * np.delete(g, d, 1).prod(1) for d in range(3)], 1)
    wz, wy, wx = np.meshgrid(w, w, w, indexing="ij")
    return N, dN, g.prod(1), db, (wx * wy * wz).ravel()


def _jacobi(n, alpha):
    """Gauss rule for the weight (1 - x)^alpha on [-1, 1] (Golub and Welsch)."""
    k = np.arange(n, dtype=float)
    s = 2.0 * k + alpha
    a = np.where(k == 0, -alpha / (alpha + 2.0), -alpha * alpha / np.maximum(s * (s + 2.0), 1e-300))
    j = np.arange(1, n, dtype=float)
    t = 2.0 * j + alpha
    b = np.sqrt(4.0 * j * (j + alpha) * j * (j + alpha) / (t * t * (t + 1.0) * (t - 1.0)))
    x, v = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    return x, 2.0 ** (alpha + 1.0) / (alpha + 1.0) * v[0] ** 2


def _tet_rule(n):
    (xu, wu), (xv, wv), (xw, ww) = _jacobi(n, 2.0), _jacobi(n, 1.0), _jacobi(n, 0.0)
    u, v, t = (a.ravel() for a in np.meshgrid(0.5 * (xu + 1), 0.5 * (xv + 1), 0.5 * (xw + 1), indexing="ij"))
    a, b, c = (a.ravel() for a in np.meshgrid(wu / 8, wv / 4, ww / 2, indexing="ij"))
    p = np.stack([u, v * (1 - u), t * (1 - u) * (1 - v)], 1)
    N = np.concatenate([1.0 - p.sum(1, keepdims=True), p], 1)
    dl = np.array([[-1.0, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]])
    dN = np.broadcast_to(dl, (p.shape[0], 4, 3)).copy()
    bub = 256.0 * N.prod(1)
    db = 256.0 * sum(np.delete(N, k, 1).prod(1)[:, None] * dl[k] for k in range(4))
    return N, dN, bub, db, a * b * c


def _element_systems(rule, X, U, beta, Up, nu, tau, f, tangent=True):
    """Element residuals (E, 4 npe), (E, 3) and blocks K_cc, K_cf, K_fc, K_ff of the weak form."""
    N, dN, b, db, w = rule
    V, P = U[..., :3], U[..., 3]
    E, npe = X.shape[:2]
    nut = (2.0 * nu).reshape(E, 1)
    J = torch.einsum("eai,qam->eqim", X, dN)
    Ji = torch.linalg.inv(J)
    om = torch.linalg.det(J) * w
    g = torch.einsum("qam,eqmj->eqaj", dN, Ji)
    d = torch.einsum("qm,eqmj->eqj", db, Ji)
    v = torch.einsum("qa,eai->eqi", N, V) + b[:, None] * beta[:, None]
    L = torch.einsum("eai,eqaj->eqij", V, g) + beta[:, None, :, None] * d[:, :, None]
    p = P @ N.T
    eye = torch.eye(3, dtype=X.dtype, device=X.device)
    src = torch.einsum("eqij,eqj->eqi", L, v) - f
    if tau:
        src = src + tau * torch.einsum("qa,eai->eqi", N, V - Up)
    src = om[..., None] * src
    sig = om[..., None, None] * (nut[..., None, None] * L - p[..., None, None] * eye)
    R = torch.zeros((E, npe, 4), dtype=X.dtype, device=X.device)
    R[..., :3] = torch.einsum("qa,eqi->eai", N, src) + torch.einsum("eqij,eqaj->eai", sig, g)
    R[..., 3] = -torch.einsum("qa,eq->ea", N, om * L.diagonal(dim1=2, dim2=3).sum(2))
    Rf = torch.einsum("q,eqi->ei", b, src) + torch.einsum("eqij,eqj->ei", sig, d)
    R = R.reshape(E, 4 * npe)
    if not tangent:
        return R, Rf
    c = torch.einsum("eqj,eqaj->eqa", v, g)
    cd = torch.einsum("eqj,eqj->eq", v, d)
    onut = nut * om
    Kcc = torch.zeros((E, npe, 4, npe, 4), dtype=X.dtype, device=X.device)
    Kcf = torch.zeros((E, npe, 4, 3), dtype=X.dtype, device=X.device)
    Kfc = torch.zeros((E, 3, npe, 4), dtype=X.dtype, device=X.device)
    NN = torch.einsum("qa,qb->qab", N, N)
    sc = (torch.einsum("qa,eqb,eq->eab", N, c, om) + torch.einsum("eqaj,eqbj,eq->eab", g, g, onut)
          + tau * torch.einsum("qab,eq->eab", NN, om))
    Kcc[:, :, :3, :, :3] = (torch.einsum("qab,eqik->eaibk", NN, om[..., None, None] * L)
                            + sc[:, :, None, :, None] * eye[None, None, :, None])
    Kcc[:, :, :3, :, 3] = -torch.einsum("eqai,qb,eq->eaib", g, N, om)
    Kcc[:, :, 3, :, :3] = -torch.einsum("qa,eqbk,eq->eabk", N, g, om)
    ob = om * b
    gd = torch.einsum("eqaj,eqj,eq->ea", g, d, onut)
    Kcf[:, :, :3] = (torch.einsum("qa,eqik->eaik", N, ob[..., None, None] * L)
                     + (torch.einsum("qa,eq->ea", N, om * cd) + gd)[..., None, None] * eye)
    Kcf[:, :, 3] = -torch.einsum("qa,eqk,eq->eak", N, d, om)
    Kfc[..., :3] = (torch.einsum("qb,eqik->eibk", N, ob[..., None, None] * L)
                    + (torch.einsum("eqb,eq->eb", c, ob) + gd + tau * torch.einsum("qb,eq->eb", N, ob))[:, None, :, None] * eye[:, None])
    Kfc[..., 3] = -torch.einsum("eqi,qb,eq->eib", d, N, om)
    Kff = (torch.einsum("eq,eqik->eik", ob * b, L)
           + (torch.einsum("eq,eq->e", ob, cd) + torch.einsum("eqj,eqj,eq->e", d, d, onut))[:, None, None] * eye)
    n = 4 * npe
    return R, Rf, Kcc.reshape(E, n, n), Kcf.reshape(E, n, 3), Kfc.reshape(E, 3, n), Kff


def exact(case, seed):
    if case["kind"].startswith("mlp"):
        return _exact_mlp(case, seed)
    # the near-null pressure modes of distorted hexahedral meshes make the solution of a linear
    # system arbitrary at the level of its conditioning; Newton's end point depends on its tolerance
    if case["kind"] == "newton" or (case["kind"] == "linear" and (case["mesh"] != "tet_cavity" or case["nx"] > 14)):
        return None
    xyz, conn, bc, u, beta, u_prev, nu, nu_e, _, _ = _workload(case, seed)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    xyz, conn, u, beta = t(xyz), t(conn).long(), t(u), t(beta)
    up = u if u_prev is None else t(u_prev)
    n_nodes, (n_elems, npe) = xyz.shape[0], conn.shape
    tau = 1.0 / case["dt"] if case.get("dt") else 0.0
    f = t(np.array(_force(case)))
    nue = torch.full((n_elems,), nu, dtype=torch.float64, device=DEV) if nu_e is None else t(nu_e)
    q = case.get("quad", 3)
    rule = [t(a) for a in (_hex_rule(q) if npe == 8 else _tet_rule(q))]
    fixed = torch.zeros(4 * n_nodes, dtype=torch.bool, device=DEV)
    fixed[t(bc.dofs)] = True
    dof = (4 * conn[:, :, None] + torch.arange(4, device=DEV)).reshape(n_elems, 4 * npe)
    rhs = torch.zeros(4 * n_nodes, dtype=torch.float64, device=DEV)
    step = 8192
    chunks = [slice(i, min(i + step, n_elems)) for i in range(0, n_elems, step)]

    def system(s, tangent=True):
        return _element_systems(rule, xyz[conn[s]], u[conn[s]], beta[s], up[conn[s]][..., :3], nue[s], tau, f, tangent)

    if case["kind"] == "residual":
        fine = torch.empty((n_elems, 3), dtype=torch.float64, device=DEV)
        for s in chunks:
            R, fine[s] = system(s, False)
            rhs.index_add_(0, dof[s].reshape(-1), R.reshape(-1))
        rhs[fixed] = 0.0
        full = torch.cat([rhs, fine.reshape(-1)])
        return {"norm": float(full.norm()), "R": full}
    # the sparsity pattern: node pairs sharing an element, sorted; 4 x 4 blocks stored row by row
    keys = torch.unique(torch.cat([torch.unique((conn[s, :, None] * n_nodes + conn[s, None, :]).reshape(-1)) for s in chunks]))
    row = keys // n_nodes
    deg = torch.bincount(row, minlength=n_nodes)
    start = torch.cumsum(deg, 0) - deg
    values = torch.zeros(16 * keys.numel(), dtype=torch.float64, device=DEV)
    four = torch.arange(4, device=DEV)
    rec = []
    for s in chunks:
        R, Rf, Kcc, Kcf, Kfc, Kff = system(s)
        sol = torch.linalg.solve(Kff, torch.cat([Kfc, Rf[..., None]], 2))
        S = Kcc - Kcf @ sol[..., :-1]
        r = R - (Kcf @ sol[..., -1:])[..., 0]
        if case["kind"] == "linear":
            rec.append(sol)
        free = ~fixed[dof[s]]
        S = S * (free[:, :, None] & free[:, None, :])
        rhs.index_add_(0, dof[s].reshape(-1), r.reshape(-1))
        pos = torch.searchsorted(keys, (conn[s, :, None] * n_nodes + conn[s, None, :]).reshape(-1)).reshape(-1, npe, npe)
        na = conn[s][:, :, None].expand(-1, npe, npe)
        base = 16 * start[na] + 4 * (pos - start[na])
        at = base[:, :, None, :, None] + (4 * deg[na])[:, :, None, :, None] * four[:, None, None] + four
        values.index_add_(0, at.reshape(-1), S.reshape(-1))
    rhs[fixed] = 0.0
    fd = torch.nonzero(fixed)[:, 0]
    nd = fd // 4
    pos = torch.searchsorted(keys, nd * n_nodes + nd)
    values[16 * start[nd] + fd % 4 * 4 * deg[nd] + 4 * (pos - start[nd]) + fd % 4] = 1.0
    if case["kind"] == "assemble":
        return {"values": values, "rhs": rhs}
    A = torch.zeros((4 * n_nodes, 4 * n_nodes), dtype=torch.float64, device=DEV)
    col = keys % n_nodes
    k = torch.arange(keys.numel(), device=DEV)
    for i in range(4):
        at = 16 * start[row] + 4 * i * deg[row] + 4 * (k - start[row])
        for j in range(4):
            A[4 * row + i, 4 * col + j] = values[at + j]
    du = torch.linalg.solve(A, -rhs)
    sol = torch.cat(rec)
    dbeta = -(sol[..., -1] + (sol[..., :-1] @ du[dof][..., None])[..., 0])
    return {"u": u + du.reshape(-1, 4), "beta": beta + dbeta}


def _exact_mlp(case, seed):
    params, x, t = _mlp_inputs(case, seed)
    p = torch.from_numpy(params).to(DEV)
    cut = [0, 1536, 1664, 18048, 18176, 18688, 18692]
    w1, b1, w2, b2, w3, b3 = (p[a:b] for a, b in zip(cut, cut[1:]))
    W = [m.bfloat16().double() for m in (w1.reshape(12, 128), w2.reshape(128, 128), w3.reshape(128, 4))]
    B = [m.double() for m in (b1, b2, b3)]
    if case["kind"] == "mlp_forward":
        return {"y": torch.cat([torch.tanh(torch.tanh(c.double() @ W[0] + B[0]) @ W[1] + B[1]) @ W[2] + B[2]
                                for c in x.split(65536)])}
    n = x.shape[0]
    loss, grad = 0.0, torch.zeros(18692, dtype=torch.float64, device=DEV)
    for c, tc in zip(x.split(65536), t.split(65536)):
        c, tc = c.double(), tc.double()
        h1 = torch.tanh(c @ W[0] + B[0])
        h2 = torch.tanh(h1 @ W[1] + B[1])
        e = h2 @ W[2] + B[2] - tc
        loss += float((e * e).sum()) / (4.0 * n)
        dy = e / (2.0 * n)
        d2 = (dy @ W[2].T) * (1.0 - h2 * h2)
        d1 = (d2 @ W[1].T) * (1.0 - h1 * h1)
        parts = (c.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ dy, dy.sum(0))
        grad += torch.cat([m.reshape(-1) for m in parts])
    return {"loss": loss, "grad": grad}
