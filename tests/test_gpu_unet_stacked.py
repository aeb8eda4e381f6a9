"""The convolution with stacked taps (up to 64 output channels) at its edges:
heights around a tile's rows, one to six channel groups, an odd K-step,
resident and streamed weights.  Bound as in test_gpu_unet_conv: one bf16
rounding (2^-8 relative) plus the cancellation of an fp32 sum."""
import numpy as np
import pytest

from oracle import unet as U
from fvv_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cout", [32, 48, 64])
@pytest.mark.parametrize("cin,h,w", [(16, 1, 5), (32, 2, 127), (40, 3, 129), (64, 4, 33), (96, 5, 130), (48, 6, 256),
                                     (176, 7, 64), (192, 9, 20)])
def test_heights_and_groups(cout, cin, h, w):
    import torch
    F = lib()
    rng = np.random.default_rng(cin + cout + h)
    x = torch.from_numpy(rng.standard_normal((2, h, w, cin)).astype(np.float32)).to(torch.bfloat16)
    wt = torch.from_numpy((rng.standard_normal((cout, 3, 3, cin)) / np.sqrt(9 * cin)).astype(np.float32)).to(torch.bfloat16)
    b = torch.from_numpy(rng.standard_normal(cout).astype(np.float32) * 0.1)
    y = torch.full((2, h, w, cout), 7.0, dtype=torch.bfloat16, device="cuda")
    F.fvv_unet_conv3x3(x.cuda(), 2, h, w, cin, wt.cuda(), b.cuda(), cout, False, None, y)
    ref = U.conv3x3(x.double().numpy(), wt.double().numpy(), b.double().numpy())
    err = np.abs(y.float().cpu().numpy() - ref)
    assert np.all(err <= 2.0 ** -8 * np.abs(ref) + 1e-3), float(err.max())


def test_relu_of_non_finite_sums():
    """A NaN sum gives 0 and an infinite one stays, as max(0, .) of the fp32 value does."""
    import torch
    F = lib()
    x = torch.zeros((1, 2, 8, 32), dtype=torch.bfloat16, device="cuda")
    x[0, 0, 2, 0] = float("inf")
    x[0, 1, 6, 0] = float("nan")
    wt = torch.zeros((32, 3, 3, 32), dtype=torch.bfloat16, device="cuda")
    wt[0, 1, 1, 0] = 1.0
    wt[1, 1, 1, 0] = -1.0
    y = torch.zeros((1, 2, 8, 32), dtype=torch.bfloat16, device="cuda")
    F.fvv_unet_conv3x3(x, 1, 2, 8, 32, wt, None, 32, True, None, y)
    g = y.float().cpu().numpy()
    assert g[0, 0, 2, 0] == np.inf and g[0, 0, 2, 1] == 0.0
    assert not np.isnan(g).any()
