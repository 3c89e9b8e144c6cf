"""Dense z-streaming kernels where a CTA's chunk of planes is long: the
straight-line steps between its ends run at every position of the unrolled
loops (ten for the smoothing, six for the regularisers)."""
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import test_regularizers_gpu as dense  # noqa: E402

pytestmark = pytest.mark.gpu

DIMS = (509, 285, 25)


def chunk(dims, resident, extra):
    """Planes a CTA takes: the split whose waves of resident CTAs of 32 x 16
    columns take the fewest steps, a chunk costing `extra` more than its planes."""
    slots = torch.cuda.get_device_properties(0).multi_processor_count * resident
    tiles = -(-dims[0] // 32) * -(-dims[1] // 16)
    best = None
    for n in range(1, (dims[2] + 3) // 4 + 1):
        zc = -(-dims[2] // n)
        cost = -(-tiles * -(-dims[2] // zc) // slots) * (zc + extra)
        if best is None or cost < best[0]:
            best = cost, zc
    return best[1]


@pytest.mark.parametrize("layout", [dense.LAYOUTS[0], dense.LAYOUTS[-1]], ids=lambda v: v[0])
def test_long_chunks(layout):
    rz = DIMS[2]
    zc = chunk(DIMS, 2, 6)  # smoothing: steps [z0 + 5, min(z1 + 2, rz) - 4)
    assert min(zc + 2, rz) - 4 - 5 >= 10
    zc = chunk(DIMS, 1, 6)  # regularisers: steps [z0 + 3, min(z1, rz) - 3)
    assert min(zc, rz) - 3 - 3 >= 6
    dense.test_smooth_parity_and_features_untouched(DIMS, layout)
    dense.test_smooth_adjoint_parity(DIMS, layout)
    dense.test_sdf_terms_parity(DIMS, layout)
