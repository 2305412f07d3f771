"""Restarted GMRES, whose next step is queued before the residual of the current one is known, against the same method
written out on the host in FP64: cycles of one step upwards, solves that end inside a cycle, on its last step and
after several cycles, and a step limit that is reached. Step counts agree to one (both sides round), and the
iterates to the accuracy that the last residual leaves: a difference of 1e-6 of the solution on these transient systems
(condition below 1e4, residuals to 1e-10)."""
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


def host_gmres(A, minv, b, rtol, maxit, restart):
    x, it, bn = np.zeros_like(b), 0, np.linalg.norm(b)
    r = b.copy()
    while it < maxit and np.linalg.norm(r) > rtol * bn:
        V, H, beta, j = [r / np.linalg.norm(r)], np.zeros((restart + 1, restart)), np.linalg.norm(r), 0
        while j < restart and it < maxit:
            w = A @ (minv @ V[j])
            for _ in range(2):
                for i, v in enumerate(V):
                    h = v @ w
                    H[i, j] += h
                    w = w - h * v
            H[j + 1, j] = np.linalg.norm(w)
            V.append(w / H[j + 1, j])
            j, it = j + 1, it + 1
            e = np.zeros(j + 1)
            e[0] = beta
            y, *_ = np.linalg.lstsq(H[:j + 1, :j], e, rcond=None)
            if np.linalg.norm(e - H[:j + 1, :j] @ y) <= rtol * bn:
                break
        x = x + minv @ (np.array(V[:j]).T @ y)
        r = b - A @ x
    return it, x


@pytest.mark.parametrize("restart", [1, 2, 3, 5, 8, 30])
@pytest.mark.parametrize("rtol,maxit", [(1e-10, 400), (1e-3, 400), (1e-10, 4)])
def test_restarts(vms, restart, rtol, maxit):
    mesh = inputs.box_mesh(4, 3, 3, hi=(4.0, 3.0, 3.0), jitter_frac=0.1, seed=5)
    u = np.random.default_rng(5).uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    ctx = vms.Context(0, 0)
    ctx.set_preconditioner(vms.PRECOND_BLOCK_JACOBI)
    dofs = np.arange(3, 4 * mesh.n_nodes, 4)  # the velocity system: well conditioned with a small time step
    ctx.mesh_upload(mesh.xyz, mesh.conn, dofs.astype(np.int64), u.reshape(-1)[dofs].copy())
    ctx.set_params(0.02, dt=0.01)
    ctx.state_upload(u, np.zeros((mesh.n_elems, 3)), u)
    ctx.assemble()
    rowptr, colidx, vals, rhs = ctx.csr_host()
    n = 4 * mesh.n_nodes
    A = sp.csr_matrix((vals, colidx, rowptr), shape=(n, n))
    minv = sp.block_diag([sp.csr_matrix(np.linalg.inv(A[4 * i:4 * i + 4, 4 * i:4 * i + 4].toarray()))
                          for i in range(mesh.n_nodes)], format="csr")
    its, x = host_gmres(A, minv, -rhs, rtol, maxit, restart)
    try:
        it, rel = ctx.solve(rtol=rtol, maxit=maxit, restart=restart, update=True)
        assert rel <= rtol and abs(it - its) <= 1, (it, its)
    except vms.VmsError as e:
        assert its >= maxit and "maxit" in str(e), (its, e)
        ctx.close()
        return
    u1, _ = ctx.state_download()
    # a count that differs by one stops at another iterate: then only the residuals bound the difference
    tol = 1e-6 if rtol < 1e-5 else 20 * rtol
    assert np.linalg.norm((u1 - u).reshape(-1) - x) <= tol * np.linalg.norm(x)
    ctx.close()
