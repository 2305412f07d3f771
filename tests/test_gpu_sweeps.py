"""The triangular sweeps of the block ILU(0) preconditioner against a plain FP64 block ILU(0) on the
host, over the shapes where their segments, chunks, batches of rows and record widths end: lines of
one row, lines shorter than a batch of rows, lines cut at 64 nodes with a remainder, partial chunks,
tetrahedra (at most eight blocks a side), and meshes in random node order (no lines; up to 26 blocks
on one side).

One GMRES step from zero with right preconditioning gives du = y M^-1 b, y from A M^-1 b in closed
form, so the state update of a solve that stops after one step shows M^-1 b itself.

Tolerances, fixed beforehand: both sides carry out the same recursion of 4x4 block products; on these
transient systems (dt = 0.01, condition numbers of the factors below 1e4) FP64 rounding gives a
relative difference below 1e4 * 2^-53 * (27 blocks * 4) ~ 1e-10. In mixed precision the factor, the
vectors and the step are FP32: below 1e4 * 2^-24 ~ 6e-4; the reference uses the FP32-rounded matrix."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vms():
    from paper_0809_4802_gb300 import build, vms as v
    build.build()
    v.load_library()
    return v


def block_ilu0(A, adj):
    """In-place block ILU(0) of {(i, j): 4x4} with sorted neighbour lists; returns the U_ii^-1."""
    dinv = {}
    for i, row in enumerate(adj):
        for k in row:
            if k >= i:
                break
            A[i, k] = A[i, k] @ dinv[k]
            for j in adj[k]:
                if j > k and (i, j) in A:
                    A[i, j] = A[i, j] - A[i, k] @ A[k, j]
        dinv[i] = np.linalg.inv(A[i, i])
    return dinv


def apply(A, dinv, adj, v):
    y = np.zeros_like(v)
    for i, row in enumerate(adj):
        y[i] = v[i] - sum((A[i, k] @ y[k] for k in row if k < i), np.zeros(4))
    z = np.zeros_like(v)
    for i in range(len(adj) - 1, -1, -1):
        z[i] = dinv[i] @ (y[i] - sum((A[i, k] @ z[k] for k in adj[i] if k > i), np.zeros(4)))
    return z


def problem(kind, dims, shuffle, seed=5):
    mesh = inputs.box_mesh(*dims, hi=tuple(float(d) for d in dims), jitter_frac=0.1, seed=seed)
    if kind == "tet":
        mesh = inputs.tet_mesh_from_lattice(mesh)
    rng = np.random.default_rng(seed)
    xyz, conn = mesh.xyz, mesh.conn
    if shuffle:
        perm = rng.permutation(mesh.n_nodes)       # new number of every node
        xyz = np.empty_like(xyz)
        xyz[perm] = mesh.xyz
        conn = np.ascontiguousarray(perm[conn].astype(np.int32))
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    return xyz, conn, u


CASES = [("hex", (1, 1, 1), False), ("hex", (3, 2, 2), False), ("hex", (4, 5, 6), False), ("hex", (66, 1, 1), False),
         ("hex", (2, 9, 3), False), ("tet", (5, 4, 3), False), ("tet", (66, 1, 1), False),
         ("hex", (4, 4, 3), True), ("tet", (4, 4, 4), True)]


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("kind,dims,shuffle", CASES, ids=[f"{k}{d[0]}x{d[1]}x{d[2]}{'s' if s else ''}" for k, d, s in CASES])
def test_one_preconditioned_step_matches_the_host(vms, kind, dims, shuffle, prec):
    xyz, conn, u = problem(kind, dims, shuffle)
    n = xyz.shape[0]
    ctx = vms.Context(0, prec)
    dofs = np.array([0, 1, 2, 3], np.int64)
    ctx.mesh_upload(xyz, conn, dofs, u.reshape(-1)[:4].copy())
    ctx.set_params(0.1, dt=0.01)
    ctx.state_upload(u, np.zeros((conn.shape[0], 3)), u)
    ctx.assemble()
    rowptr, colidx, vals, rhs = ctx.csr_host()
    vals = vals.astype(np.float64)
    adj, A = [], {}
    for i in range(n):
        lo, hi = rowptr[4 * i], rowptr[4 * i + 1]
        adj.append([int(c) // 4 for c in colidx[lo:hi:4]])
        for t, j in enumerate(adj[i]):
            A[i, j] = np.array([vals[rowptr[4 * i + r] + 4 * t:rowptr[4 * i + r] + 4 * t + 4] for r in range(4)])
    S = dict(A)
    dinv = block_ilu0(A, adj)
    b = -rhs.reshape(n, 4)
    beta = np.linalg.norm(b)
    z = apply(A, dinv, adj, b / beta)
    w = np.zeros_like(z)
    for (i, j), blk in S.items():
        w[i] += blk @ z[j]
    h0 = np.sum(w * b) / beta
    h1 = np.linalg.norm(w - h0 * b / beta)
    ref = beta * h0 / (h0 * h0 + h1 * h1) * z
    assert h1 / np.hypot(h0, h1) < 0.999          # one step meets the tolerance below
    ctx.solve(rtol=0.999, maxit=1, restart=1, update=True)
    u1, _ = ctx.state_download()
    err = np.linalg.norm((u1 - u) - ref) / np.linalg.norm(ref)
    assert err < (1e-10 if prec == 0 else 6e-4), err
    ctx.close()
