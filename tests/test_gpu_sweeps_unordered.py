"""The ILU(0) factorisation and sweeps on numberings without grid lines and with lines in random order, against the plain
FP64 block ILU(0) of test_gpu_sweeps, at the sizes where the kernels' forms change: levels of more rows than the GPU has SMs
(one warp per row) and fewer, segments of one row (no rings of copies), hexahedra (up to 26 blocks on one side of a
row) and tetrahedra, and chunks whose far neighbours exceed the limit, so that a chunk takes fewer lines.

As there, one GMRES step from zero shows M^-1 b itself; the tolerances are those derived there (1e-10 in FP64, 6e-4 in
mixed precision)."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs
from test_gpu_sweeps import apply, block_ilu0

pytestmark = pytest.mark.gpu


def numbering(kind, mesh, dims):
    rng = np.random.default_rng(9)
    if kind == "random":
        return rng.permutation(mesh.n_nodes)
    # lines along x keep their order inside, the lines themselves are shuffled
    lines = mesh.n_nodes // (dims[0] + 1)
    return (rng.permutation(lines)[:, None] * (dims[0] + 1) + np.arange(dims[0] + 1)).reshape(-1)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("tet,dims,order", [(False, (6, 6, 6), "random"), (False, (19, 19, 19), "random"),
                                            (True, (16, 15, 15), "random"), (False, (63, 7, 7), "lines"),
                                            (True, (63, 7, 7), "lines")],
                         ids=["hex7", "hex20", "tet17", "hex64 lines", "tet64 lines"])
def test_one_preconditioned_step_matches_the_host(vms, tet, dims, order, prec):
    mesh = inputs.box_mesh(*dims, hi=tuple(float(d) for d in dims), jitter_frac=0.1, seed=5)
    if tet:
        mesh = inputs.tet_mesh_from_lattice(mesh)
    n = mesh.n_nodes
    perm = numbering(order, mesh, dims)
    xyz = np.empty_like(mesh.xyz)
    xyz[perm] = mesh.xyz
    conn = np.ascontiguousarray(perm[mesh.conn].astype(np.int32))
    u = np.random.default_rng(5).uniform(-0.5, 0.5, (n, 4))
    ctx = vms.Context(0, prec)
    ctx.mesh_upload(xyz, conn, np.array([0, 1, 2, 3], np.int64), u.reshape(-1)[:4].copy())
    ctx.set_params(0.1, dt=0.01)
    ctx.state_upload(u, np.zeros((conn.shape[0], 3)), u)
    ctx.assemble()
    rowptr, colidx, vals, rhs = ctx.csr_host()
    vals = vals.astype(np.float64)
    adj, A = [], {}
    for i in range(n):
        rows = [vals[rowptr[4 * i + r]:rowptr[4 * i + r + 1]].reshape(-1, 4) for r in range(4)]
        adj.append([int(c) // 4 for c in colidx[rowptr[4 * i]:rowptr[4 * i + 1]:4]])
        blocks = np.stack(rows, 1)
        for t, j in enumerate(adj[i]):
            A[i, j] = blocks[t]
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
    assert h1 / np.hypot(h0, h1) < 0.999
    ctx.solve(rtol=0.999, maxit=1, restart=1, update=True)
    u1, _ = ctx.state_download()
    err = np.linalg.norm((u1 - u) - ref) / np.linalg.norm(ref)
    assert err < (1e-10 if prec == 0 else 6e-4), err
    ctx.close()
