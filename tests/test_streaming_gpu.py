"""The z-streaming grid kernels at the sizes where they can go wrong: one node
short of, at and past a tile's edge (32 x 16 columns), z split over several
CTAs, and brick columns walked eight bricks at a time (enough stored bricks for
that rule), each against the oracle at the tolerances of the general cases.
"""
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import test_regularizers_gpu as dense  # noqa: E402
import test_sparse_gpu as sparse  # noqa: E402

pytestmark = pytest.mark.gpu

EDGES = [(31, 15, 7), (32, 16, 8), (33, 17, 9), (65, 33, 130), (3, 2, 70)]
LONG = (96, 96, 2240)  # 5040 bricks, about half of them stored


@pytest.mark.parametrize("dims", EDGES)
@pytest.mark.parametrize("layout", [dense.LAYOUTS[0], dense.LAYOUTS[-1]], ids=lambda v: v[0])
def test_dense_tile_edges(dims, layout):
    dense.test_smooth_parity_and_features_untouched(dims, layout)
    dense.test_smooth_adjoint_parity(dims, layout)
    dense.test_sdf_terms_parity(dims, layout)


def test_long_brick_columns():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert int(sparse.random_bricks(LONG, sum(LONG)).sum()) >= 16 * sms
    sparse.test_sparse_smoothing_matches_the_full_grid(LONG)
    sparse.test_sparse_sdf_regularizers_match_the_full_grid(LONG)


def test_long_brick_columns_transposed():
    """<G x, y> = <x, G^T y> with empty = 0 on the same brick mask, where both
    operators walk eight bricks at a time (the forward is pinned above)."""
    import paper_2412_10084_gb300 as ps
    keep = torch.as_tensor(sparse.random_bricks(LONG, 9))
    n = int(keep.sum())
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    x, y = (torch.randn(n, 16, 16, 16, generator=gen, device="cuda") for _ in range(2))
    zero = torch.zeros(n, 16, 16, 16, 3, device="cuda")
    sc = ps.sparse_scene(keep, torch.zeros_like(x), zero, torch.zeros(2, 2, 2, 9, 4),
                         torch.zeros(ps.mlp_param_count(10, 32)), LONG, (0, 0, 0), (1, 1, 20), 3,
                         32, empty_sdf=0.0)
    gd, _, _ = sc.descs(3)
    w = ps.table_words(gd)
    ps.sdf_smooth(gd, x, sc.grid)
    gx = sc.grid.view(-1)[w:].view(-1, 4)[:, 0].double()
    gg = sc.grad_buffers()[0]
    gg.view(-1)[w:].view(-1, 4)[:, 0] = y.view(-1)
    gty = torch.zeros_like(x)
    ps.sdf_smooth_adjoint(gd, gg, gty, accumulate=False)
    a = float((gx * y.view(-1).double()).sum())
    b = float((x.view(-1).double() * gty.view(-1).double()).sum())
    scale = float((gx.abs() * y.view(-1).abs().double()).sum())
    # each output of either side is a sum of 125 products in FP32 (relative
    # rounding of a pass at most 5 half-units, three passes: 15 * 2^-24)
    assert abs(a - b) <= 2 * 15 * 2.0 ** -24 * 5 * scale
