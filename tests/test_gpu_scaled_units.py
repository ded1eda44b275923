"""The compression does not depend on the unit of length.

A power of two in the data scales every float32 value exactly, so that a compression
takes the same steps at any scale whose entries, and the sums of their squares over a
row, are in float32's range: the same ranks, pivots and entry counts, and factors
scaled by it.  The squared norms, their products and the stopping tests of a block go
beyond that range.

* dense faces: a separable tensor with entries around 1 and around 2^57 (1.4e17).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(40, 40)])
def test_separable_scale(g3, M, N):
    ctx = g3.Context(0)
    rng = np.random.default_rng(M)
    R, Ku = 6, 16
    a, b, c = (rng.standard_normal((R, k)) + 1j * rng.standard_normal((R, k)) for k in (M, N, Ku))
    a *= 10.0 ** -np.arange(R)[:, None]
    fas = [g3.aca3_compress_separable(ctx, a * s, b, c, prec="mixed", eps3=1e-3) for s in (1.0, 2.0 ** 57)]
    (s0, s1), (b0, b1) = [f.stats() for f in fas], [f.block(0, M, N, Ku) for f in fas]
    assert (s0["dense_crosses"] > 0) == (M * N <= 48 * 48)
    assert s0["entries"] == s1["entries"] and s0["crosses"] == s1["crosses"] and s0["crosses"] > 1
    assert np.array_equal(b0["piv"], b1["piv"])
    assert np.array_equal(b0["f"], b1["f"])
