"""The gradient of the warm-start network at the row counts where its tile changes (16, 32 or 64 rows, one round
of CTAs each) and around partial tiles, with and without an index list, read back to host memory and into device
memory. Tolerances: those of the network's other gradient tests, 1e-4 of a block's largest entry (two-term BF16
products, FP32 sums) and 1e-5 of the loss."""
import ctypes

import numpy as np
import pytest

from oracle import warmstart as ows
from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def net():
    from paper_0809_4802_gb300 import build, vms
    build.build()
    vms.load_library()
    m = vms.Mlp(0)
    m.set_stream(torch.cuda.current_stream().cuda_stream)
    m.set_params(inputs.mlp_init(7))
    yield m
    m.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, "16", "16+1", "32", "32+1", "64+5"])
@pytest.mark.parametrize("listed", [False, True])
def test_gradient_at_the_tile_edges(net, n, listed):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if isinstance(n, str):
        r, _, more = n.partition("+")
        n = int(r) * sms + int(more or 0)
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n + 3, 12)).astype(np.float32)
    T = rng.normal(size=(n + 3, 4)).astype(np.float32)
    idx = rng.permutation(n + 3)[:n].astype(np.int32)
    x, t = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    rows = torch.from_numpy(idx).cuda() if listed else None
    loss, g = net.grad(x, t, rows=rows, n=None if listed else n)
    at = idx if listed else np.arange(n)
    p = net.get_params(stored=False)
    lref, gref = ows.loss_and_grad(ows.stored(p), X[at].astype(np.float64), T[at].astype(np.float64))
    assert abs(loss - lref) <= 1e-5 * lref
    a, b = ows.unpack(g.astype(np.float64)), ows.unpack(ows.pack(gref))
    for k in b:
        assert np.abs(a[k] - b[k]).max() <= 1e-4 * np.abs(b[k]).max(), k
    # into device memory, with and without the loss
    d = torch.full((len(g) + 1,), 7.0, device="cuda")
    out = ctypes.c_double()
    rp = rows.data_ptr() if listed else None
    for lp in (ctypes.byref(out), None):
        assert net.lib.vms_mlp_grad(net.h, n, rp, x.data_ptr(), t.data_ptr(), lp, d.data_ptr()) == 0
        assert np.abs(d[:-1].cpu().numpy() - g).max() <= 1e-5 * np.abs(g).max() and d[-1] == 7.0
    assert abs(out.value - loss) <= 1e-10 * loss
