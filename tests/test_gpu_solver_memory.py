"""What a mixed solve allocates: the FP64 row records of the ILU(0) sweeps (two per node of at least 8 places of 132
bytes) come with the first solve whose FP32 refinement stalls, not with every mixed solve."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_fp64_sweep_records_come_on_first_use(vms):
    mesh = inputs.box_mesh(24, 24, 24, hi=(24.0, 24.0, 24.0), jitter_frac=0.1, seed=5)
    u = np.random.default_rng(5).uniform(-0.5, 0.5, (mesh.n_nodes, 4))
    ctx = vms.Context(0, vms.PREC_MIXED)
    dofs = np.arange(3, 4 * mesh.n_nodes, 4)  # the velocity system: well conditioned with a small time step
    ctx.mesh_upload(mesh.xyz, mesh.conn, dofs.astype(np.int64), u.reshape(-1)[dofs].copy())
    ctx.set_params(0.02, dt=0.01)
    ctx.state_upload(u, np.zeros((mesh.n_elems, 3)), u)
    ctx.assemble()
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    ctx.solve(rtol=1e-3, maxit=3000, restart=150, update=False)
    one = free()
    ctx.solve(rtol=1e-3, maxit=3000, restart=150, update=False)
    assert free() == one
    with pytest.raises(vms.VmsError) as ei:       # below what FP64 can reach: the refinement stalls
        ctx.solve(rtol=1e-18, maxit=3000, restart=150, update=False)
    assert ei.value.code == vms.ERR_KRYLOV_MAXIT
    records = 2 * 8 * 132 * mesh.n_nodes
    kept_vectors = 150 * 8 * 4 * mesh.n_nodes    # of the flexible form
    assert one - free() >= records + kept_vectors
    ctx.close()
