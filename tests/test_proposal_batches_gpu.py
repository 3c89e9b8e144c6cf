"""The proposal's training kernels at the batch and sample counts where they can
go wrong: CTAs with one ray, one short of and past a full CTA, more rays than the
resident CTAs take at once; chunks of 32 samples cut short."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import oracle  # noqa: E402
import test_proposal_gpu as base  # noqa: E402
from helpers import rel_err_tensor  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2412_10084_gb300 as ps


@pytest.mark.parametrize("B", [8, 16])
@pytest.mark.parametrize("n", [1, 127, 129, 40000])
def test_backward_batches(B, n):
    sc, o, d = base.scene_and_rays(n_rays=1500, seed_offset=5 + B)
    prm = base.proposal_params(seed=8, logit_scale=1.0, B=B)
    res, thr = (16, 16, 16), base.threshold_f32(sc)
    m = oracle.Model.from_scene(sc)
    prop = oracle.Proposal(oracle.occupancy(m, res, thr), prm, n_bins=B, mix=base.MIX, theta=0.2)
    hist = oracle.weight_histogram(m, o, d, 64.0, 64, B).astype(np.float32)
    # rays with mass, at least 1e-4 from a ReLU kink (both precisions switch alike)
    keep = (oracle.proposal_forward(m, prop, o, d, 8)["margin"] > 1e-4) & (hist.sum(1) >= 1e-2)
    pick = np.resize(np.nonzero(keep)[0], n)
    o, d, hist = o[pick], d[pick], hist[pick]
    g_ref, loss_ref = oracle.proposal_backward(m, prop, o, d, hist.astype(np.float64), 1e-3,
                                               1.0 / n)
    scene = ps.Scene.from_host(sc)
    occ = ps.occupancy_build(scene, res, thr)
    desc = ps.proposal_desc(res, n_bins=B, mix=base.MIX, theta=0.2)
    grad, loss = ps.proposal_backward(scene, desc, base.dev(prm), occ, base.dev(o), base.dev(d),
                                      base.dev(hist), 1e-3, 1.0 / n)
    assert np.max(np.abs(loss.cpu().numpy() - loss_ref) / np.maximum(loss_ref, 1e-2)) <= 1e-5
    # the bound of the general case (FP32 sums over the rays)
    assert rel_err_tensor(grad.cpu().numpy(), g_ref) <= 1e-4


@pytest.mark.parametrize("N,B", [(1, 1), (31, 31), (32, 1), (33, 11), (65, 5), (256, 32)])
def test_histogram_sample_counts(N, B):
    sc, o, d = base.scene_and_rays(n_rays=300, seed_offset=70 + N)
    hist = ps.weight_histogram(ps.Scene.from_host(sc), base.dev(o), base.dev(d),
                               ps.render_params(64.0, N), B)
    ref = oracle.weight_histogram(oracle.Model.from_scene(sc), o, d, 64.0, N, B)
    assert np.max(np.abs(hist.cpu().numpy() - ref)) <= 2e-6
