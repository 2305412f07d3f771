"""The warm-start network's forward pass with infinite parameters (a network whose training has run away): a hidden
unit whose bias or input weight is infinite is saturated at +-1, as tanh of the sum in 64 bits is, and not a NaN of
the products' BF16 terms (a zero lower term times an infinity). Inputs are BF16 numbers (their lower terms are zero)
and ones that are not; where the sum itself is NaN (0 times infinity, infinity minus infinity) the outputs are.
Tolerance as in test_gpu_mlp_forward: 28 x 2^-23 x 8 / |y| < 3e-5 of the largest output."""
import numpy as np
import pytest

from paper_0809_4802_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

B1, W2, B2, W3, B3 = 1536, 1664, 18048, 18176, 18688


@pytest.mark.parametrize("params", [{B1: np.inf}, {B1 + 127: -np.inf}, {B2: np.inf}, {B2 + 64: -np.inf}, {0: np.inf},
                                    {128 * 11 + 5: -np.inf}, {0: np.inf, B1: -np.inf}, {B1: np.nan}, {7: np.nan}],
                         ids=["b1", "-b1", "b2", "-b2", "w1", "-w1", "w1-b1", "nan b1", "nan w1"])
def test_infinite_parameters_saturate(vms, params):
    net = vms.Mlp(0)
    net.set_stream(torch.cuda.current_stream().cuda_stream)
    p = inputs.mlp_init(5).astype(np.float32)
    for at, v in params.items():
        p[at] = v
    net.set_params(p)
    x = torch.randn((200, 12), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    x[:100] = torch.round(x[:100]) + 0.5   # BF16 numbers, none of them zero
    x[150] = 0.0
    y = torch.empty((200, 4), device="cuda")
    net.forward(x, y)
    q = torch.from_numpy(net.get_params(stored=True).astype(np.float64)).cuda()
    h = torch.tanh((x.double()[:, :, None] * q[:B1].view(1, 12, 128)).sum(1) + q[B1:W2])
    h = torch.tanh(h @ q[W2:B2].view(128, 128) + q[B2:W3])
    ref = h @ q[W3:B3].view(128, 4) + q[B3:]
    nan = torch.isnan(ref)
    assert torch.equal(torch.isnan(y), nan)
    if not nan.all():
        assert (y.double() - ref)[~nan].abs().max() < 3e-5 * ref[~nan].abs().max()
    net.close()
