"""The frequency after an overruled stop is the same in every run.

Two separable terms on disjoint rows and columns: the second lives at the frequencies
5..12 alone, with one value, so that the crosses of the first end in a stop which the
samples overrule with equal residual energies at 5..12.  Their sums over the samples
have to be equal too, whatever the order in which threads come by, so that the smallest
index is taken.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [40, 96])   # dense faces, low-rank faces
def test_next_frequency_after_an_overruled_stop(g3, n, prec):
    ctx = g3.Context(0)
    rng = np.random.default_rng(n)
    Ku, h = 24, n // 2
    a, b = (rng.standard_normal((3, n)) + 1j * rng.standard_normal((3, n)) for _ in range(2))
    for x in (a, b):
        x[0, h:] = 0
        x[1, :h] = 0
    a[2] *= 1e-5
    c = np.zeros((3, Ku), dtype=complex)
    c[0] = 1.0
    c[1, 5:13] = 0.5
    c[2] = rng.standard_normal(Ku)   # keeps the second face from vanishing
    c[2, 5:13] = c[2, 5]
    seen = set()
    for _ in range(30):
        fa = g3.aca3_compress_separable(ctx, a, b, c, prec=prec, eps3=1e-3)
        assert fa.stats()["stop_check_overrides"] >= 1
        seen.add(tuple(fa.block(0, n, n, Ku)["piv"][:, 2].tolist()))
    assert len(seen) == 1, seen
    assert 5 in next(iter(seen)) and not set(range(6, 13)) & set(next(iter(seen)))
