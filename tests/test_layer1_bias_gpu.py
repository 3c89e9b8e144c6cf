"""Layer 1's bias is an FP32 addition in the render: biases past FP16's range
count in full where the sum with W1 x is in range again."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import synth  # noqa: E402
from helpers import oracle_forward  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2412_10084_gb300 as ps


# (feature, W1, b1): layer 1 sums to 36000 and to 34000
@pytest.mark.parametrize("feature,w,b", [(1.0, -30000.0, 66000.0), (2.0, 50000.0, -66000.0)])
def test_bias_past_half_range(feature, w, b):
    sc = synth.make_scene("sphere64", dims=(24, 24, 24), probe_dims=(6, 6, 6))
    rays = synth.make_rays("sphere64", n_rays=256)
    sc.feat[...] = feature
    W = sc.width
    n_in = (sc.mlp.size - (W + W * W + W + 3 * W + 3)) // W
    mlp = sc.mlp.copy()
    w1 = mlp[:W * n_in].reshape(W, n_in)
    w1[...] = 0.0
    w1[:, 0] = w
    mlp[W * n_in:W * n_in + W] = b
    mlp[-(3 * W + 3):-3] *= 1e-5  # layer 3 brings the units back to the colour scale
    sc.mlp = mlp
    rgb = ps.render_forward(ps.Scene.from_host(sc), torch.as_tensor(rays.o, device="cuda"),
                            torch.as_tensor(rays.d, device="cuda"),
                            ps.render_params(64.0, 64, 0, sc.n_fresnel))[0].cpu().numpy()
    ref = oracle_forward(sc, rays.o, rays.d, 64.0, 64)
    assert (ref["wsum"] > 0.5).sum() > 20
    # A unit is about 1e-6 off (22-bit operands, FP32 sums of terms up to three
    # times the unit): 36000 x 1e-6 x 16 units x |W2| of 0.2 is 0.12 in a unit of
    # layer 2, x 16 x |W3| of 3e-6 is 6e-6 in a logit, 1.5e-6 in a colour; the
    # opacities add their 1e-6.  Without the units the colours are 0.1 off.
    assert np.max(np.abs(rgb - ref["rgb"])) <= 1e-5
