"""The residual at the element counts where its split changes, against the FP64 oracle: a lane per line of
the Gauss rule (small meshes, and what is left after whole rounds of a thread per element) for the rules
of 8, 27 and 64 points, which take 8, 3 and 2 elements per warp, with counts that leave a warp partly
empty; through the element records, the assembled residual vector and the assembly itself (in mixed
precision the fused kernel). Tolerance: both sides sum the same terms in FP64 in another order, a few
hundred terms each: 1e-12 of the largest entry."""
import numpy as np
import pytest

import oracle
from oracle import Params
from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vms():
    from paper_0809_4802_gb300 import build, vms as v
    build.build()
    v.load_library()
    return v


# one element; partly empty warps for every rule; a partial round behind one whole round on 152 SMs
@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 1, 1), (5, 5, 7), (31, 19, 37)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("quad", [2, 3, 4])
@pytest.mark.parametrize("dt,f", [(0.0, (0.0, 0.0, 0.0)), (0.0, (0.3, -0.2, 0.5)), (0.01, (0.0, 0.0, 0.0)),
                                  (0.01, (0.3, -0.2, 0.5))], ids=["steady", "force", "transient", "both"])
def test_residual_split_matches_oracle(vms, dims, quad, dt, f):
    mesh = inputs.box_mesh(*dims, hi=tuple(0.5 * d for d in dims), jitter_frac=0.15, seed=4)
    n = mesh.n_elems
    rng = np.random.default_rng(9)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    beta = rng.uniform(-0.1, 0.1, (n, 3))
    up = u + rng.uniform(-0.01, 0.01, u.shape)
    p = Params(nu=0.02, dt=dt, f=f, quad_order=quad)
    X, U, _, Up = oracle.gather(mesh.conn, mesh.xyz, u, beta, up if dt else None)
    k = oracle.element_residual_only(X, U, beta, p, Up)
    Rcp, Rf = oracle.pack_residual(k)
    dofs = np.array([1, 4 * mesh.n_nodes - 4], np.int64)
    for prec in (0, 1):
        ctx = vms.Context(0, prec)
        ctx.mesh_upload(mesh.xyz, mesh.conn, dofs, u.reshape(-1)[dofs].copy())
        ctx.set_params(p.nu, p.visc_factor, p.dt, p.f, p.bubble_scale, p.quad_order)
        ctx.state_upload(u, beta, up if dt else None)
        first = 0 if n < 1000 else n - 500
        got = ctx.element_matrices(first, n - first)
        assert np.abs(got["Rcp"] - Rcp[first:]).max() < 1e-12 * np.abs(Rcp).max()
        assert np.abs(got["Rf"] - Rf[first:]).max() < 1e-12 * np.abs(Rf).max()
        ref = oracle.residual_vector(mesh.conn, mesh.n_nodes, k, dofs)
        norm, r = ctx.residual(want_vector=True)
        assert np.abs(r - ref).max() < 1e-12 * np.abs(ref).max()
        assert abs(norm - np.linalg.norm(ref)) < 1e-12 * norm
        # the assembly: r_e = R_cp - K_cf K_ff^-1 R_f on its own residual records; K_cf and K_ff are
        # FP32 in mixed precision (1e-5, as for the assembled system elsewhere)
        ctx.assemble()
        rhs = ctx.csr_host()[3]
        if n < 1000:
            Kcc, Kcf, Kfc, Kff, _, _ = oracle.pack_element(oracle.element_kernel(X, U, beta, p, Up))
            _, re, _, _ = oracle.condense(Kcc, Kcf, Kfc, Kff, Rcp, Rf)
            want = oracle.assemble_vector(mesh.conn, mesh.n_nodes, re)
            want[dofs] = 0.0
            assert np.abs(rhs - want).max() < (1e-10, 1e-5)[prec] * np.abs(want).max()
        ctx.close()
