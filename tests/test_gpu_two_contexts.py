"""Two contexts and two networks on their own streams and host threads at once: the Arnoldi step is a cooperative launch
that needs every SM, the sweeps' blocks wait for each other, and the network's blocks share tensor memory, so each has
to make room for the other's. The results are those of the same calls one after the other, bit for bit (coloured
scatter: the order of every sum is fixed; the networks' gradients are not compared)."""
import threading

import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_two_threads_get_what_one_gets(vms):
    work, streams = [], [torch.cuda.Stream() for _ in range(2)]
    for t, (n, prec) in enumerate(((14, 0), (18, 1))):
        wl = inputs.cavity_workload(n, re=100.0, jitter_frac=0.1, state="noise", seed=n)
        ctx = vms.Context(0, prec)
        ctx.set_stream(streams[t].cuda_stream)
        ctx.mesh_upload(wl.mesh.xyz, wl.mesh.conn, wl.bc.dofs, wl.bc.vals)
        ctx.set_params(wl.nu, scatter_mode=vms.SCATTER_COLOUR)
        net = vms.Mlp(0)
        net.set_stream(streams[t].cuda_stream)
        net.set_params(inputs.mlp_init(t).astype(np.float32))
        x = torch.randn((60000, 12), generator=torch.Generator(device="cuda").manual_seed(t), device="cuda")
        work.append((ctx, wl, net, x, torch.empty((60000, 4), device="cuda")))
    torch.cuda.synchronize()

    def run(t, out, repeats):
        ctx, wl, net, x, y = work[t]
        for _ in range(repeats):
            ctx.state_upload(wl.u, wl.beta)
            ctx.assemble()
            net.forward(x, y)
            it = ctx.solve(rtol=1e-4, maxit=3000, restart=100, update=True)
            streams[t].synchronize()
            out.append((it, ctx.state_download()[0].tobytes(), y.cpu().numpy().tobytes()))

    alone = [[], []]
    for t in range(2):
        run(t, alone[t], 1)
    both = [[], []]
    threads = [threading.Thread(target=run, args=(t, both[t], 6)) for t in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join(timeout=120)
        assert not th.is_alive()
    for t in range(2):
        assert len(both[t]) == 6 and all(r == alone[t][0] for r in both[t])
        work[t][0].close()
        work[t][2].close()
