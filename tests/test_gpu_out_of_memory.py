"""A solve that runs out of device memory at any of its allocations reports VMS_ERR_OUT_OF_MEMORY and keeps no part of
what it was allocating: with memory back, the same context solves the same system. The rest of the device memory is
held by one tensor, so that the allocations of the solver's vectors, of the ILU(0) pattern and of its factor fail one
after the other as a little more is left free."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_a_solve_without_memory_leaves_nothing_half_made(vms, prec):
    wl = inputs.cavity_workload(24, re=100.0, jitter_frac=0.1, state="noise", seed=4)
    failed = 0
    for left in (4, 12, 24, 40, 60, 80, 100, 120, 140, 160, 200, 240, 300):
        ctx = vms.Context(0, prec)
        ctx.mesh_upload(wl.mesh.xyz, wl.mesh.conn, wl.bc.dofs, wl.bc.vals)
        ctx.set_params(wl.nu)
        ctx.state_upload(wl.u, wl.beta)
        ctx.assemble()
        solve = lambda: ctx.solve(rtol=1e-3, maxit=3000, restart=30, update=False)  # noqa: E731
        torch.cuda.empty_cache()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - left * MB, dtype=torch.uint8, device="cuda")
        for _ in range(2):          # the second meets what the first left
            try:
                solve()
            except vms.VmsError as e:
                assert e.code == vms.ERR_OUT_OF_MEMORY, (left, str(e))
                failed += 1
        del hold
        torch.cuda.empty_cache()
        it, rel = solve()
        assert rel <= 1e-3
        ctx.close()
    assert failed >= 8
