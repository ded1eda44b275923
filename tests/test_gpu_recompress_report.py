"""A float32 face whose recompression breaks down is reported.

One value of a separable tensor's factor is not a number, so that every face holds a row
of them.  The block ends (its faces have no finite pivot or fewer crosses), and the
status bit and the counter of recompressions that broke down say so, as in float64.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
RECOMPRESSION = 1 << 2


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, None])
def test_breakdown_is_reported(g3, bad, prec):
    ctx = g3.Context(0)
    rng = np.random.default_rng(1)
    a, b, c = (rng.standard_normal((4, k)) + 1j * rng.standard_normal((4, k)) for k in (80, 70, 9))
    if bad is not None:
        a[1, 40] = bad
    st = g3.aca3_compress_separable(ctx, a, b, c, prec=prec, eps3=1e-4, dense_face_max=-1).stats()
    assert (st["status_bits"] & RECOMPRESSION != 0) == (bad is not None)
    assert (st["recompress_fallbacks"] > 0) == (bad is not None)
