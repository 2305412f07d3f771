"""The warm-start network's forward pass (tcgen05 tiles of 128 rows, two CTAs per SM) against FP64 on the stored
weights: row counts around a tile and around a whole round of CTAs, X and Y 16-byte aligned or not, and
infinities, NaN and the largest values in X. Tolerance: 128 FP32 products per sum, each of the 28 partial sums
rounded or cut off at 2^-23 of a sum of |terms| below 8: 28 x 2^-23 x 8 / |y| < 3e-5 of the largest output."""
import numpy as np
import pytest

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
    p = inputs.mlp_init(5)
    p[1536:1664] = np.linspace(-0.3, 0.3, 128)
    p[18048:18176] = np.linspace(0.2, -0.2, 128)
    p[18688:] = (0.1, -0.2, 0.3, 0.05)
    m.set_params(p.astype(np.float32))
    yield m
    m.close()


def reference(m, x):
    p = torch.from_numpy(m.get_params(stored=True).astype(np.float64)).to(x.device)
    h = torch.tanh(x.double() @ p[:1536].view(12, 128) + p[1536:1664])
    h = torch.tanh(h @ p[1664:18048].view(128, 128) + p[18048:18176])
    return h @ p[18176:18688].view(128, 4) + p[18688:]


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 1000, "round", "round+1", "2 rounds+65"])
@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "unaligned"])
def test_forward_matches_fp64(net, n, shift):
    full = 2 * torch.cuda.get_device_properties(0).multi_processor_count * 128
    n = {"round": full, "round+1": full + 1, "2 rounds+65": 2 * full + 65}.get(n, n)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(12 * n + shift, generator=g, device="cuda")[shift:].view(n, 12)
    y = torch.full((4 * n + shift + 4,), 7.0, device="cuda")
    out = y[shift:shift + 4 * n].view(n, 4)
    assert net.lib.vms_mlp_forward(net.h, n, x.data_ptr(), out.data_ptr()) == 0
    ref = reference(net, x)
    assert (out.double() - ref).abs().max() < 3e-5 * ref.abs().max()
    assert torch.all(y[:shift] == 7.0) and torch.all(y[shift + 4 * n:] == 7.0)  # nothing beside the rows


def test_forward_special_values(net):
    x = torch.randn((300, 12), device="cuda")
    special = [float("inf"), -float("inf"), 3.4e38, -3.4e38, 1e-38, 1e-42, -0.0, 1e20]
    for i, v in enumerate(special):
        x[7 * i, i] = v
    x[150, 3] = float("nan")
    x[200, 0], x[200, 1] = float("inf"), float("inf")
    y = torch.empty((300, 4), device="cuda")
    net.forward(x, y)
    ref = reference(net, x)
    nan = torch.isnan(ref)
    assert nan[150].all()
    assert torch.equal(torch.isnan(y), nan)
    assert (y.double() - ref)[~nan].abs().max() < 3e-5 * ref[~nan].abs().max()
