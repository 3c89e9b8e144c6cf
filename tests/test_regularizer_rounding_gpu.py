"""The regularisers' divisions and square roots are FP32's correctly rounded ones,
and gradients of s down to nothing follow the FP64 oracle."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import synth  # noqa: E402
import test_regularizers_gpu as dense  # noqa: E402
from helpers import rel_err_tensor  # noqa: E402
from oracle import regularizers as R  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2412_10084_gb300 as ps


def terms(s, s_hat, bmin, bmax, lam):
    """(d s, loss) of the SDF terms on a BF16-feature grid (s in its own array)."""
    dims = s.shape[::-1]
    gd, values, _ = dense.make_grid(dims, bmin, bmax, s, ps.BF16, ps.FEAT_NODES, 1)
    grad = torch.zeros(ps.grid_bytes(gd)[1] // 4, dtype=torch.float32, device="cuda")
    loss = torch.zeros(4, dtype=torch.float32, device="cuda")
    ps.grid_regularizers(gd, dense.dev(s_hat), values, grad,
                         torch.zeros(s.shape, dtype=torch.float32, device="cuda"), *lam, loss=loss)
    return (ps.unpack_grid(gd, grad, which=ps.GRID_GRAD)[0].cpu().numpy(),
            loss.cpu().numpy())


def test_voxel_weight_is_correctly_rounded():
    """L_sdf with s - s_hat = 1: d s is twice the weight 1 / (1 + 5 |s|)."""
    g = synth.rng(3)
    s = (g.integers(-2 ** 20, 2 ** 20, size=(24, 33, 40)) * 2.0 ** -20).astype(np.float32)
    s_hat = (s.astype(np.float64) - 1.0).astype(np.float32)
    keep = s.astype(np.float64) - s_hat.astype(np.float64) == 1.0  # s_hat exact
    assert keep.mean() > 0.4
    ds, _ = terms(s, s_hat, (0, 0, 0), (1, 1, 1), (1.0, 0.0, 0.0))
    den = (1.0 + 5.0 * np.abs(s.astype(np.float64))).astype(np.float32)
    w = (1.0 / den.astype(np.float64)).astype(np.float32)
    assert np.array_equal(ds[keep], (2.0 * w)[keep])


@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e15])
def test_gradient_norm_and_normal(scale):
    """One interior node with the gradient (a, b, 0): L_Eik shows the norm, and d s
    of the x-neighbours the normal, for norms around 1 and on both sides of those
    where the kernel changes its way (1e-8 and 1e15)."""
    g = synth.rng(4)
    for a, b in (scale * g.uniform(0.5, 1.1, size=(96, 2))).astype(np.float32):
        step = np.array([-1, 0, 1], np.float32)
        s = np.zeros((3, 3, 3), np.float32)
        s[1, 1] += a * step
        s[1, :, 1] += b * step
        ds, loss = terms(s, s, (-1, -1, -1), (1, 1, 1), (0.0, 1.0, 0.0))  # spacing 1
        # the kernel's sum of squares: a a rounded, then one fused step
        gg = np.float32(np.float64(a * a) + np.float64(b) * np.float64(b))
        norm = np.sqrt(gg)
        assert norm.dtype == np.float32
        e = norm - np.float32(1.0)
        assert loss[1] == e * e, (a, b)
        # d s = e n / h: the normal's reciprocal is a unit in the last place off,
        # the products half a unit each
        n = float(a) / np.sqrt(float(a) ** 2 + float(b) ** 2)
        assert abs(ds[1, 1, 2] / (float(e) * n) - 1.0) <= 2.0 ** -21, (a, b)
        assert ds[1, 1, 0] == -ds[1, 1, 2]


@pytest.mark.parametrize("slope", [1e-6, 1e-8, 3e-9, 1e-12, 0.0])
def test_nearly_flat_fields(slope):
    """Slopes on both sides of the norms that FP32 tells from their
    regularised form, a flat half and a step."""
    dims = (37, 20, 18)
    g = synth.rng(9)
    s = (slope * np.cumsum(1.0 + 0.2 * g.normal(size=dims[::-1]), axis=2)).astype(np.float32)
    s[:, :, 20:] = 0.0
    bmin, bmax = (0.0, 0.0, 0.0), tuple(float(d - 1) for d in dims)  # spacing 1
    for lam in ((0.0, 1.0, 0.0), (0.0, 0.0, 1.0)):
        ds, loss = terms(s, s, bmin, bmax, lam)
        vals, ref, _ = R.sdf_terms(s, s, R.spacing(dims, bmin, bmax), *lam)
        for part in (slice(0, 17), slice(17, None)):  # the step's gradients are far larger
            assert rel_err_tensor(ds[..., part], ref[..., part]) <= dense.GRAD_RTOL
        for i, name in ((1, "eik"), (2, "normal")):
            assert abs(float(loss[i]) - vals[name]) <= dense.LOSS_RTOL * max(abs(vals[name]), 1.0)
