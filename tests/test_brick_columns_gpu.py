"""How many bricks a CTA of the sparse grid passes walks: the results do not
depend on it, and a grid with fewer stored bricks is not the slower one."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import synth  # noqa: E402
import test_regularizers_gpu as dense  # noqa: E402
from helpers import rel_err_tensor  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2412_10084_gb300 as ps

LAM = (1.0, 0.1, 0.02)


def bricks_per_cta(dims):
    """The rule: doubled up to 8 as long as 12 CTAs per SM remain."""
    b, seg = [d // 16 for d in dims], 1
    enough = 12 * torch.cuda.get_device_properties(0).multi_processor_count
    while seg < 8 and seg < b[2] and b[0] * b[1] * -(-b[2] // (2 * seg)) >= enough:
        seg *= 2
    return seg


def sparse_grid(dims, keep, sdf):
    box_max = tuple(float(d - 1) for d in dims)  # spacing 1
    return ps.sparse_scene(keep, sdf, torch.zeros(*sdf.shape, 3, device="cuda"),
                           torch.zeros(2, 2, 2, 9, 4), torch.zeros(ps.mlp_param_count(10, 32)),
                           dims, (0, 0, 0), box_max, 3, 32, empty_sdf=0.5)


@pytest.mark.parametrize("far,seg", [((256, 256, 256), 2), ((384, 384, 256), 4),
                                     ((768, 768, 256), 8)])
def test_same_results_in_a_larger_grid(far, seg):
    """The same bricks in a grid where a CTA walks one, and in the corner of one
    where it walks `seg`.  No brick is stored next to the small grid's far faces
    in x and y, so the stencils see the same nodes."""
    near = (64, 64, 256)
    assert bricks_per_cta(near) == 1 and bricks_per_cta(far) == seg
    g = synth.rng(5)
    corner = g.uniform(size=(16, 3, 3)) < 0.6
    n = int(corner.sum())
    s = torch.as_tensor(g.uniform(0.2, 0.8, size=(n, 16, 16, 16)), dtype=torch.float32,
                        device="cuda")
    out = []
    for dims in (near, far):
        keep = np.zeros([d // 16 for d in dims[::-1]], bool)
        keep[:, :3, :3] = corner
        sc = sparse_grid(dims, torch.as_tensor(keep), s)
        gd, _, _ = sc.descs(3)
        w = ps.table_words(gd)
        grad = sc.grad_buffers()[0]
        d_hat, loss = torch.zeros_like(s), torch.zeros(4, device="cuda")
        ps.grid_regularizers(gd, s + 0.01, sc.grid, grad, d_hat, *LAM, loss=loss)
        back = torch.ones_like(s)
        ps.sdf_smooth_adjoint(gd, grad, back, accumulate=True)
        ps.sdf_smooth(gd, s, sc.grid)
        out.append([t.cpu().numpy() for t in (sc.grid.view(-1)[w:], grad.view(-1)[w:], d_hat,
                                              back, loss)])
    a, b = out
    assert np.max(np.abs(a[0] - b[0])) <= dense.SMOOTH_ATOL
    for x, y in zip(a[1:4], b[1:4]):
        assert rel_err_tensor(y, x) <= dense.GRAD_RTOL
    assert np.all(np.abs(a[4] - b[4]) <= dense.LOSS_RTOL * np.abs(a[4]))


def test_few_bricks_in_a_large_grid():
    """1024^3 nodes: the passes over 300 stored bricks take no longer than over
    3000 (with one brick per CTA they took three times as long)."""
    dims = (1024, 1024, 1024)
    times = []
    for n in (300, 3000):
        keep = torch.zeros(64, 64, 64, dtype=torch.bool)
        keep.view(-1)[torch.as_tensor(synth.rng(1).permutation(64 ** 3)[:n])] = True
        s = torch.full((n, 16, 16, 16), 0.1, device="cuda")
        sc = sparse_grid(dims, keep, s)
        gd, _, _ = sc.descs(3)
        grad, d_hat = sc.grad_buffers()[0], torch.zeros_like(s)
        best = float("inf")
        for _ in range(5):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            ps.sdf_smooth(gd, s, sc.grid)
            ps.grid_regularizers(gd, s, sc.grid, grad, d_hat, *LAM)
            ps.sdf_smooth_adjoint(gd, grad, d_hat)
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end))
        times.append(best)
    assert times[0] <= 1.1 * times[1], times
