"""The matrix-vector product with 32 and with 16 lanes per node (small and larger meshes; rows of 8 to 27 blocks and
rows of a tetrahedral mesh), with vectors that are 16-byte aligned and not, against the assembled matrix in FP64. The
same at most 108 products summed in FP64 in another order: 1e-13 of the sum of magnitudes."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vms():
    from paper_0809_4802_gb300 import build, vms as v
    build.build()
    v.load_library()
    return v


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind,dims", [("hex", (1, 1, 1)), ("hex", (5, 3, 2)), ("hex", (17, 17, 16)), ("tet", (4, 3, 2)),
                                       ("tet", (17, 17, 16))])
def test_apply(vms, kind, dims, shift, prec):
    mesh = inputs.box_mesh(*dims, hi=tuple(float(d) for d in dims), jitter_frac=0.1, seed=2)
    if kind == "tet":
        mesh = inputs.tet_mesh_from_lattice(mesh)
    rng = np.random.default_rng(3)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    ctx = vms.Context(0, prec)
    dofs = np.array([0, 3], np.int64)
    ctx.mesh_upload(mesh.xyz, mesh.conn, dofs, u.reshape(-1)[dofs].copy())
    ctx.set_params(0.02)
    ctx.state_upload(u)
    ctx.assemble()
    rowptr, colidx, values, _ = ctx.csr_host()
    n = 4 * mesh.n_nodes
    A = sp.csr_matrix((values.astype(np.float64), colidx, rowptr), shape=(n, n))
    x = torch.randn(n + shift, dtype=torch.float64, device="cuda")[shift:]
    y = torch.full((n + shift + 1,), 7.0, dtype=torch.float64, device="cuda")
    ctx.apply(x, y[shift:shift + n])
    torch.cuda.synchronize()
    xh = x.cpu().numpy()
    assert np.all(np.abs(y[shift:shift + n].cpu().numpy() - A @ xh) <= 1e-13 * (abs(A) @ np.abs(xh)))
    assert torch.all(y[:shift] == 7.0) and y[-1] == 7.0
    ctx.close()
