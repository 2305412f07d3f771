"""The triangular sweeps give up, not only the factorisation before them: the factor is made and kept at the default
wait limit, then one poll per wait ends the waits of the sweeps' rows, far neighbours and copies at every place where
they can be (lines that fit the copies in flight and longer ones, no lines at all). Each such solve returns
VMS_ERR_TIMEOUT, no copy is left in flight behind its block, and the same context then solves the kept system in as
many steps as before (the factor is made again: an error discards it)."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("dims,tet,shuffle", [((8, 8, 8), False, False), ((20, 9, 8), False, False), ((12, 12, 12), True, False),
                                              ((9, 9, 9), False, True)], ids=["lines9", "lines21", "tet13", "shuffled"])
def test_sweeps_that_give_up_are_reported_and_recover(vms, dims, tet, shuffle, prec):
    mesh = inputs.box_mesh(*dims, hi=tuple(float(d) for d in dims), jitter_frac=0.1, seed=3)
    if tet:
        mesh = inputs.tet_mesh_from_lattice(mesh)
    xyz, conn = mesh.xyz, mesh.conn
    rng = np.random.default_rng(3)
    if shuffle:
        perm = rng.permutation(mesh.n_nodes)
        xyz = np.empty_like(mesh.xyz)
        xyz[perm] = mesh.xyz
        conn = np.ascontiguousarray(perm[mesh.conn].astype(np.int32))
    u = rng.uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    ctx = vms.Context(0, prec)
    ctx.mesh_upload(xyz, conn, np.array([0, 1, 2, 3], np.int64), u.reshape(-1)[:4].copy())
    ctx.set_params(0.1, dt=0.01)
    ctx.state_upload(u, np.zeros((conn.shape[0], 3)), u)
    ctx.assemble()
    solve = lambda: ctx.solve(rtol=1e-5, maxit=3000, restart=150, update=False)  # noqa: E731
    it, rel = solve()
    assert rel <= 1e-5
    for _ in range(3):
        ctx.set_wait_limit(1)
        with pytest.raises(vms.VmsError) as ei:
            solve()
        assert ei.value.code == vms.ERR_TIMEOUT
        ctx.set_wait_limit(0)
        it2, rel2 = solve()
        assert rel2 <= 1e-5 and abs(it2 - it) <= 1
    ctx.close()
