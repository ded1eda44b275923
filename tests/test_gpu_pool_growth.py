"""A block that needs many times its pool estimate is compressed.

Full-rank tensors: every face reaches the rank cap and every frequency takes a cross, 7.4
and 3.3 times what the estimate of such a block reserves.  The spill rounds have to grow
the pool until it fits, and the result is that of a pool that was large enough.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Ku,prec", [(100, 40, "mixed"), (100, 40, "fp64"), (40, 40, "mixed")])
def test_block_beyond_its_estimate(g3, n, Ku, prec):
    rng = np.random.default_rng(n)
    a, b, c = (rng.standard_normal((80, k)) + 1j * rng.standard_normal((80, k)) for k in (n, n, Ku))
    fas = [g3.aca3_compress_separable(g3.Context(0), a, b, c, prec=prec, eps3=1e-6, pool_factor=p) for p in (0.0, 100.0)]
    (s, t), (x, y) = [f.stats() for f in fas], [f.block(0, n, n, Ku) for f in fas]
    assert s["spilled_blocks"] > 0 and t["spilled_blocks"] == 0
    assert s["crosses"] == t["crosses"] == Ku
    assert np.array_equal(x["piv"], y["piv"]) and np.array_equal(x["f"], y["f"])
    assert all(np.array_equal(u, v) for u, v in zip(x["U"], y["U"]))
