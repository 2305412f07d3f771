"""Elements of very small edges in FP64: the element matrices of a mesh scaled by s = 2^-k with viscosity nu are s^2
times those of the mesh as it is with viscosity nu / s (the weak form's terms all scale alike), and a power of two
scales every operation exactly as long as no intermediate underflows. det J ~ s^3 is a normal number down to edges of
about 1e-102, and so must all that is formed on the way be. Tolerance 1e-13 of the largest entry: the same roundings on
both sides (an intermediate of the size of a product of two cofactors would lose 1e-11 at edges of 1e-78)."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0, 200, 259, 282, 316])
@pytest.mark.parametrize("quad", [2, 3])
@pytest.mark.parametrize("tet", [False, True], ids=["hex", "tet"])
def test_element_matrices_scale(vms, tet, quad, k):
    hexm = inputs.cavity_mesh(2, 0.1, 1)
    bc = inputs.cavity_bc(hexm)
    mesh = inputs.tet_mesh_from_lattice(hexm) if tet else hexm
    rng = np.random.default_rng(1)
    u, beta = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4)), rng.uniform(-0.1, 0.1, (mesh.n_elems, 3))
    s, got = 2.0 ** -k, []
    for xyz, nu in ((mesh.xyz, 0.125 / s), (mesh.xyz * s, 0.125)):
        ctx = vms.Context(0, 0)
        ctx.mesh_upload(np.ascontiguousarray(xyz), mesh.conn, bc.dofs, bc.vals)
        ctx.set_params(nu, quad_order=quad)
        ctx.state_upload(u, beta)
        ctx.assemble()
        got.append(ctx.element_matrices(0, mesh.n_elems))
        ctx.close()
    for key, ref in got[0].items():
        a = got[1][key] / s / s
        assert np.abs(a - ref).max() <= 1e-13 * np.abs(ref).max(), key
