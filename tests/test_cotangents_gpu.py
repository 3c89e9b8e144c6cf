"""Autograd of the render where a loss uses only some of its outputs: the others
come to the backward without a cotangent."""
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import synth  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2412_10084_gb300 as ps


@pytest.mark.parametrize("used", [(1,), (2,), (1, 2), (0, 2)])
def test_missing_cotangents_count_as_zero(used):
    sc = synth.make_scene("sphere64", dims=(24, 24, 24), probe_dims=(6, 6, 6))
    rays = synth.make_rays("sphere64", n_rays=300)
    scene = ps.Scene.from_host(sc)
    params = ps.render_params(64.0, 64, 0, sc.n_fresnel)
    o, d = (torch.as_tensor(a, device="cuda") for a in (rays.o, rays.d))
    leaves = [t.clone().requires_grad_(True) for t in (scene.grid, scene.probes, scene.mlp)]
    out = ps.RenderFunction.apply(*leaves, o, d, None, scene, params)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    weights = [torch.randn(t.shape, generator=g, device="cuda") for t in out]
    sum((out[i] * weights[i]).sum() for i in used).backward()
    logT = ps.render_forward(scene, o, d, params)[3]
    full = [w if i in used else torch.zeros_like(w) for i, w in enumerate(weights)]
    ref = ps.render_backward(scene, o, d, params, full[0], logT, d_depth=full[1], d_wsum=full[2])
    for leaf, r in zip(leaves, ref):
        # the same sums, reduced in another order
        assert float((leaf.grad - r).abs().max()) <= 1e-5 * max(float(r.abs().max()), 1e-30)
    assert float(leaves[0].grad.abs().max()) > 0.0
