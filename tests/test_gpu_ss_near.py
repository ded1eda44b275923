"""Near-field entries of element pairs with a common vertex, edge or panel on an irregular
closed mesh: the float32 Sauter-Schwab kernels (points in float-float, pair list built on the
device) against the float64 ones, pair by pair."""
from __future__ import annotations

import numpy as np
import pytest

from inputs import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["slp", "hyp", "adj"])
@pytest.mark.parametrize("shape", ["sphere", "cube"])
def test_float32_singular_pairs(kernel, shape):
    import paper_2312_11219_gb300 as g3
    v, t = meshes.icosphere(2) if shape == "sphere" else meshes.cube(3)
    rng = np.random.default_rng(7)
    v = v * np.array([1.0, 0.5, 2.0]) + 0.01 * rng.standard_normal(v.shape)   # no two panels alike
    ctx = g3.Context(0)
    T = g3.build_cluster_tree(ctx, v, t, 16, 1.0)
    if kernel != "slp":
        T = g3.build_p1_tree(ctx, T)
    F = g3.g3_freqs_gcq(ctx, 22, 0.05, 0.15)      # 11 unique frequencies: not a multiple of the warps
    Ku = F.info()[1]
    near = {p: g3.assemble_near(ctx, T, F, kernel, "galerkin4x4", p) for p in ("fp64", "mixed")}
    info = T.get()
    d = 3 if kernel != "slp" else 1
    perm = info["perm"][::d] // d      # element of each cluster position
    shared = (t[perm][:, None, :, None] == t[perm][None, :, None, :]).any(axis=(2, 3))
    seen = 0
    for b, (rb, re, cb, ce, far) in enumerate(info["blocks"]):
        if far:
            continue
        A, B = (near[p].block(b, re - rb, ce - cb, Ku) for p in ("mixed", "fp64"))
        # the local 3 x 3 (1 x 1) entries of each element pair; float32 entries within 3e-5 of the
        # pair's largest one (the bound of the float32 entries elsewhere in this suite)
        q = lambda X: X.reshape(Ku, (re - rb) // d, d, (ce - cb) // d, d).transpose(0, 1, 3, 2, 4).reshape(  # noqa: E731
            Ku, (re - rb) // d, (ce - cb) // d, d * d)
        a, r = q(A), q(B)
        size = np.abs(r).max(axis=3, keepdims=True)
        if kernel == "adj":     # exactly singular on a flat panel: against the block's entries
            size = np.maximum(size, 1e-3 * np.abs(r).max(axis=(1, 2, 3), keepdims=True))
        m = shared[rb // d:re // d, cb // d:ce // d]
        assert (np.abs(a - r) <= 3e-5 * size)[:, m].all(), (b, float((np.abs(a - r) / size)[:, m].max()))
        seen += int(m.sum())
    assert seen == int(shared.sum())
