"""The last kernel of an assembly, y = K_ff^-1 R_f and r_e = R_cp - K_cf y with eight threads per element, and
the constrained rows it sets, at element counts around a warp (4 elements) and a block (16) and with every
kind of constraint count. r_e against the same product of the element blocks the library hands out (FP32
in mixed precision, read exactly), in FP64: a few roundings of the terms, 1e-13 of the largest entry times
the 3 x 3 solve's condition (below 100): 1e-11. The assembled right-hand side against the sum of r_e: 1e-11
in FP64; in mixed precision K_cf of the assembly is summed in another order in FP32: 1e-5."""
import numpy as np
import pytest

import oracle
from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vms():
    from paper_0809_4802_gb300 import build, vms as v
    build.build()
    v.load_library()
    return v


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("scatter", [0, 1])
@pytest.mark.parametrize("n,n_dir", [(1, 0), (2, 1), (3, 128), (4, 40), (15, 129), (16, 0), (17, 1), (65, 300)])
def test_finish(vms, prec, scatter, n, n_dir):
    mesh = inputs.box_mesh(n, 1, 1, hi=(0.5 * n, 0.5, 0.5), jitter_frac=0.15, seed=2)
    rng = np.random.default_rng(n)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    beta = rng.uniform(-0.1, 0.1, (n, 3))
    n_dir = min(n_dir, 4 * mesh.n_nodes - 1)
    dofs = np.sort(rng.choice(4 * mesh.n_nodes, n_dir, replace=False)).astype(np.int64)
    ctx = vms.Context(0, prec)
    ctx.mesh_upload(mesh.xyz, mesh.conn, dofs, u.reshape(-1)[dofs].copy())
    ctx.set_params(0.02, dt=0.01, f=(0.1, 0.2, -0.3), scatter_mode=scatter)
    ctx.state_upload(u, beta, u + rng.uniform(-0.01, 0.01, u.shape))
    got = ctx.element_matrices(0, n)
    y = np.linalg.solve(got["Kff"], got["Rf"][:, :, None])[:, :, 0]
    r = got["Rcp"] - np.einsum("eck,ek->ec", got["Kcf"], y)
    assert np.abs(got["r"] - r).max() < 1e-11 * np.abs(r).max()
    ctx.assemble()
    rowptr, colidx, values, rhs = ctx.csr_host()
    want = oracle.assemble_vector(mesh.conn, mesh.n_nodes, r)
    want[dofs] = 0.0
    assert np.abs(rhs - want).max() < (1e-11, 1e-5)[prec] * np.abs(want).max()
    assert np.all(rhs[dofs] == 0.0)
    for d in dofs:  # a unit diagonal in an otherwise zero row
        row = slice(rowptr[d], rowptr[d + 1])
        assert np.array_equal(values[row], (colidx[row] == d).astype(values.dtype))
    ctx.close()
