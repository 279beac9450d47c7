"""The fused inference kernel's operand blocks (64 and 32 K-elements wide), column groups of zero to four 16-column
chunks and its two accumulators in turn: bit for bit the layer-by-layer result, and the same for rows that hold
infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,width", [(32, 32), (64, 32), (32, 96), (64, 160), (64, 192), (32, 224), (64, 224), (32, 256)])
@pytest.mark.parametrize("n", [1, 128, 129, 128 * 152 * 2 + 1])
def test_fused_shapes_equal_layer_by_layer(d_in, width, n):
    import torch
    from paper_2411_07920_gb300 import swcs as S
    rng = np.random.default_rng(n + d_in + width)
    net = S.Mlp(d_in, width)
    net.set_params(rng.normal(0.0, 0.2, size=width * d_in + width * width + 3 * width + 1).astype(np.float32))
    x = rng.normal(size=(n, d_in)).astype(np.float32)
    if n > 1:
        x[0, 3], x[n // 2, 0], x[n - 1, d_in - 1] = np.inf, np.nan, -np.inf
    d_x = torch.from_numpy(x).cuda().to(torch.bfloat16).view(torch.int16)
    y_ref = torch.empty(n, dtype=torch.float32, device="cuda")
    y = torch.full((n,), 7.0, dtype=torch.float32, device="cuda")
    net.forward_dev(d_x, y_ref)
    net.predict_dev(d_x, y)
    net.sync()
    assert torch.allclose(y, y_ref, rtol=0.0, atol=0.0, equal_nan=True)
    net.close()
