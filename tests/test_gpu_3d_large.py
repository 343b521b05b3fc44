"""Three-dimensional lattices whose two state buffers exceed the 126 MB L2, where
the slices and column launches take other segment heights: the same bits as
the per-axis passes."""
import numpy as np
import pytest

from paper_2604_21128_gb300 import qla

pytestmark = pytest.mark.gpu


# sites above 126e6 / (2 buffers x 6 planes x bytes): 2.63e6 FP32, 1.31e6 FP64;
# ragged in every direction
@pytest.mark.parametrize("shape,precision", [((162, 150, 110), "fp32"), ((258, 101, 103), "fp32"),
                                             ((118, 110, 103), "fp64")])
def test_segments_beyond_the_l2_agree_bitwise(shape, precision):
    nx, ny, nz = shape
    assert 12 * nx * ny * nz * (8 if precision == "fp64" else 4) > 126e6
    rng = np.random.default_rng(nx)
    n = 1.0 + rng.random((nz, ny, nx))
    n[: nz // 2] = 1.5
    q0 = rng.standard_normal((6, nz, ny, nx))
    out = []
    for kernel in ("passes", "slices"):
        with qla.Grid3(nx, ny, nz, 1.0, precision) as g:
            g.set_step_kernel(kernel)
            g.set_medium(n)
            g.set_state(q0)
            g.step(5)
            out.append(g.get_state())
    assert np.array_equal(out[0], out[1])
