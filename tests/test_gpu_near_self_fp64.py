"""Float64 self entries of the single layer are as accurate as their points summed one by one.

The near field's moment series and the point-by-point routine of g3_entries, frequencies
from |s| rmax = 0.05 to 30 in several directions, right-angled and stretched triangles.
Each of the two is within 1e-15 of the 72-point sum in more digits (series up to |s| rmax
= 3.5: 7.7e-16), so that they agree to 2e-15.
"""
import numpy as np
import pytest

from inputs import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [(1.0, 1.0, 1.0), (1.0, 0.3, 1.7)])
def test_float64_self_entries(g3, stretch):
    v, t = meshes.cube(3)
    v = v * np.array(stretch)
    P = v[t]
    rmax = float(np.linalg.norm(P - P.mean(1, keepdims=True), axis=2).max())
    s = np.concatenate([np.geomspace(0.05, 30.0, 24) / rmax * np.exp(1j * p) for p in (0.0, 0.6, 1.2, 1.55)])
    ctx = g3.Context(0)
    T = g3.build_cluster_tree(ctx, v, t, 8, 1.0)
    F = g3.g3_freqs_from_array(ctx, s)
    Ku, E = F.info()[1], t.shape[0]
    tg = T.get()
    ids = np.arange(E)
    ref = g3.g3_entries(ctx, T, F, "slp", ids, ids, np.arange(s.size), "fp64")
    nf = g3.assemble_near(ctx, T, F, "slp", prec="fp64")
    seen = 0
    for b, (rb, re, cb, ce, far) in enumerate(tg["blocks"]):
        if far or rb != cb:
            continue
        d = np.einsum("kii->ik", nf.block(b, re - rb, ce - cb, Ku))
        want = ref[tg["perm"][rb:re]]
        assert (np.abs(d - want) / np.abs(want)).max() <= 2e-15
        seen += re - rb
    assert seen == E
