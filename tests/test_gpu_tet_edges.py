"""The tetrahedral assembly where it can go wrong: element counts around a warp (8) and a block (16), every
combination of time step and body force, and results narrowed to FP32 over its whole range, subnormal numbers
included (elements of size 1 down to 1e-19, where some entries leave the normal range). Blocks against the FP64
oracle: 1e-10 of the largest entry, as for the hexahedron. Mixed CSR values against the FP64 element matrices:
each term is rounded once (2^-24) and so is each of at most 24 sums, of the terms' magnitudes: 25 x 2^-24 of the sum of
magnitudes, plus one subnormal step (1.4e-45) each."""
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


def tet_box(dims, h, seed=3):
    return inputs.tet_mesh_from_lattice(inputs.box_mesh(*dims, hi=tuple(h * d for d in dims), jitter_frac=0.1, seed=seed))


@pytest.mark.parametrize("count", [1, 7, 8, 9, 15, 16, 17, 33])
@pytest.mark.parametrize("dt,f", [(0.0, (0.0, 0.0, 0.0)), (0.0, (0.3, -0.2, 0.5)), (0.01, (0.0, 0.0, 0.0)), (0.01, (0.3, -0.2, 0.5))],
                         ids=["steady", "force", "transient", "both"])
def test_tet_blocks_at_partial_warps(vms, count, dt, f):
    mesh = tet_box((4, 2, 2), 0.5)
    rng = np.random.default_rng(count)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    beta = rng.uniform(-0.1, 0.1, (mesh.n_elems, 3))
    up = u + rng.uniform(-0.01, 0.01, u.shape)
    p = Params(nu=0.02, dt=dt, f=f)
    p.element = "tet"
    first = mesh.n_elems - count
    conn = mesh.conn[first:]
    X, U, _, Up = oracle.gather(conn, mesh.xyz, u, beta[first:], up if dt else None)
    Kcc, Kcf, Kfc, Kff, Rcp, Rf = oracle.pack_element(oracle.element_kernel(X, U, beta[first:], p, Up))
    S, r, _, _ = oracle.condense(Kcc, Kcf, Kfc, Kff, Rcp, Rf)
    ctx = vms.Context(0, 1)
    ctx.mesh_upload(mesh.xyz, mesh.conn, np.array([0], np.int64), u.reshape(-1)[:1].copy())
    ctx.set_params(p.nu, p.visc_factor, p.dt, p.f, p.bubble_scale, p.quad_order)
    ctx.state_upload(u, beta, up if dt else None)
    got = ctx.element_matrices(first, count)
    for key, ref in dict(Kcc=Kcc, Kcf=Kcf, Kfc=Kfc, Kff=Kff, Rcp=Rcp, Rf=Rf, S=S, r=r).items():
        assert np.abs(got[key] - ref).max() < 1e-10 * np.abs(ref).max(), key
    ctx.close()


@pytest.mark.parametrize("h", [1.0, 1e-6, 1e-12, 1e-17, 1e-19])
def test_tet_results_in_fp32(vms, h):
    mesh = tet_box((2, 2, 1), h)
    rng = np.random.default_rng(1)
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    beta = rng.uniform(-0.1, 0.1, (mesh.n_elems, 3))
    ctx = vms.Context(0, 1)
    dofs = np.array([5], np.int64)
    ctx.mesh_upload(mesh.xyz, mesh.conn, dofs, u.reshape(-1)[dofs].copy())
    ctx.set_params(0.02, scatter_mode=1)  # by colours: FP32 atomic adds flush subnormal numbers to zero
    ctx.state_upload(u, beta)
    S = ctx.element_matrices(0, mesh.n_elems)["S"]
    ctx.assemble()
    rowptr, colidx, values, _ = ctx.csr_host()
    A, _ = oracle.assemble(mesh.conn, mesh.n_nodes, S, np.zeros(S.shape[:2]))
    B, _ = oracle.assemble(mesh.conn, mesh.n_nodes, np.abs(S), np.zeros(S.shape[:2]))
    rows = np.repeat(np.arange(4 * mesh.n_nodes), np.diff(rowptr))
    want, size = A.toarray()[rows, colidx], B.toarray()[rows, colidx]
    free = (rows != 5) & (colidx != 5)
    assert np.all(np.abs(values - want)[free] <= 25 * 2.0 ** -24 * size[free] + 25 * 1.4e-45)
    if h == 1e-19:  # the case reaches the subnormal numbers
        assert np.any((np.abs(S) > 0) & (np.abs(S) < 1.2e-38))
    ctx.close()
