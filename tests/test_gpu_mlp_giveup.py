"""A forward pass of the warm-start network that gives up waiting for the tensor cores: with one poll per wait it cannot
see its products finished, with tiles after it (the next tile's products are in flight when it gives up) or without.
Every row is NaN or right, the next call reports VMS_ERR_TIMEOUT once, and at the default limit the same network
computes again. Tolerance as in test_gpu_mlp_forward."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 1000, 200001])
def test_forward_that_gives_up_is_reported(vms, n):
    net = vms.Mlp(0)
    net.set_stream(torch.cuda.current_stream().cuda_stream)
    net.set_params(inputs.mlp_init(5).astype(np.float32))
    p = torch.from_numpy(net.get_params(stored=True).astype(np.float64)).cuda()
    x = torch.randn((n, 12), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    h = torch.tanh(x.double() @ p[:1536].view(12, 128) + p[1536:1664])
    h = torch.tanh(h @ p[1664:18048].view(128, 128) + p[18048:18176])
    ref = h @ p[18176:18688].view(128, 4) + p[18688:]
    y = torch.zeros((n, 4), device="cuda")
    for call in ("forward", "get_params", "adam"):
        net.set_wait_limit(1)
        net.forward(x, y)
        torch.cuda.synchronize()
        net.set_wait_limit(0)
        nan = torch.isnan(y)
        assert nan.any() and torch.equal(nan, nan[:, :1].expand(-1, 4))
        if not nan.all():
            assert (y.double() - ref)[~nan].abs().max() < 3e-5 * ref.abs().max()
        with pytest.raises(vms.VmsError) as ei:
            {"forward": lambda: net.forward(x, y), "get_params": net.get_params, "adam": lambda: net.adam(1e-3)}[call]()
        assert ei.value.code == vms.ERR_TIMEOUT
        net.forward(x, y)
        torch.cuda.synchronize()
        assert (y.double() - ref).abs().max() < 3e-5 * ref.abs().max()
    with pytest.raises(vms.VmsError) as ei:
        net.set_wait_limit(-1)
    assert ei.value.code == vms.ERR_INVALID_ARG
    net.close()
