"""The Arnoldi step in one launch (ortho_kernel) against GMRES written out on the host in FP64, with the
same block-Jacobi preconditioner, at the sizes where its split changes: one block and a partial warp of
rows (8 nodes), one block's most rows (128 nodes) and just more than one block (144 and 150 nodes),
with bases from one vector to more than the eight a warp takes at a time and than 32 warps' worth.

Both sides take the same steps, so in FP64 they need the same number of iterations up to one (the
residual that ends the solve may lie within rounding of the tolerance) and the solutions differ by
no more than the two residuals allow: 2 rtol cond(A), cond(A) taken from the matrix."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vms():
    from paper_0809_4802_gb300 import build, vms as v
    build.build()
    v.load_library()
    return v


def host_gmres(A, minv, b, rtol, maxit):
    n = b.size
    beta = np.linalg.norm(b)
    V = [b / beta]
    H = np.zeros((maxit + 1, maxit))
    for j in range(maxit):
        w = A @ (minv @ V[j])
        Q = np.array(V)
        h = Q @ w
        w = w - Q.T @ h
        h2 = Q @ w
        w = w - Q.T @ h2
        H[:j + 1, j] = h + h2
        H[j + 1, j] = np.linalg.norm(w)
        V.append(w / H[j + 1, j])
        e = np.zeros(j + 2)
        e[0] = beta
        y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
        if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= rtol * beta:
            return j + 1, minv @ (np.array(V[:-1]).T @ y)
    raise AssertionError("host GMRES did not converge")


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 3, 7), (3, 3, 8), (4, 4, 5)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_gmres_takes_the_host_s_steps(vms, dims, prec):
    mesh = inputs.box_mesh(*dims, hi=tuple(float(d) for d in dims), jitter_frac=0.1, seed=3)
    rng = np.random.default_rng(3)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    ctx = vms.Context(0, prec)
    ctx.set_preconditioner(vms.PRECOND_BLOCK_JACOBI)
    ctx.mesh_upload(mesh.xyz, mesh.conn, np.array([0, 1, 2, 3], np.int64), u.reshape(-1)[:4].copy())
    ctx.set_params(0.1, dt=0.05)
    ctx.state_upload(u, np.zeros((mesh.n_elems, 3)), u)
    ctx.assemble()
    rowptr, colidx, vals, rhs = ctx.csr_host()
    n = 4 * mesh.n_nodes
    A = sp.csr_matrix((vals.astype(np.float64), colidx, rowptr), shape=(n, n))
    minv = sp.block_diag([sp.csr_matrix(np.linalg.inv(A[4 * i:4 * i + 4, 4 * i:4 * i + 4].toarray()))
                          for i in range(mesh.n_nodes)], format="csr")
    rtol = 1e-8
    its, x = host_gmres(A, minv, -rhs, rtol, 400)
    it, rel = ctx.solve(rtol=rtol, maxit=400, restart=400, update=True)
    u1, _ = ctx.state_download()
    assert rel <= rtol
    if prec == 0:
        assert abs(it - its) <= 1, (it, its)
    cond = np.linalg.cond(A.toarray())
    err = np.linalg.norm((u1 - u).reshape(-1) - x) / np.linalg.norm(x)
    assert err <= 2 * rtol * cond, (err, cond)
    ctx.close()
