"""The compression does not depend on the unit of length.

A power of two in the data scales every float32 value exactly, so that a compression
takes the same steps at any scale whose entries, and the sums of their squares over a
row, are in float32's range: the same ranks, pivots and entry counts, and factors
scaled by it.  The squared norms, their products and the stopping tests of a block go
beyond that range.

* dense faces and on-demand low-rank faces: a separable tensor with entries around 1
  and around 2^57 (1.4e17) and 2^55;
* low-rank faces with and without the dense residual working face: the single layer on
  the cube at 2^60 times the size, frequencies 2^-60 (entries up to 1e15).
"""
import numpy as np
import pytest

from inputs import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,e", [(40, 40, 57), (120, 100, 55)])
def test_separable_scale(g3, M, N, e):
    ctx = g3.Context(0)
    rng = np.random.default_rng(M)
    R, Ku = 6, 16
    a, b, c = (rng.standard_normal((R, k)) + 1j * rng.standard_normal((R, k)) for k in (M, N, Ku))
    a *= 10.0 ** -np.arange(R)[:, None]
    fas = [g3.aca3_compress_separable(ctx, a * s, b, c, prec="mixed", eps3=1e-3) for s in (1.0, 2.0 ** e)]
    (s0, s1), (b0, b1) = [f.stats() for f in fas], [f.block(0, M, N, Ku) for f in fas]
    assert (s0["dense_crosses"] > 0) == (M * N <= 48 * 48)
    assert s0["entries"] == s1["entries"] and s0["crosses"] == s1["crosses"] and s0["crosses"] > 1
    assert np.array_equal(b0["piv"], b1["piv"])
    assert np.array_equal(b0["f"], b1["f"])


@pytest.mark.parametrize("residual_face_max", [0, -1])
def test_single_layer_scale(g3, residual_face_max):
    import torch
    ctx = g3.Context(0)
    w = workloads.get("cube768")
    W = torch.from_numpy(workloads.densities(w.E, w.freq.K, 3).T.copy()).to("cuda", torch.complex64).t()
    out = []
    for s in (1.0, 2.0 ** 60):
        T = g3.build_cluster_tree(ctx, w.verts * s, w.tris, w.leaf, w.eta)
        F = g3.g3_freqs_bdf2(ctx, w.freq.K, w.freq.lam, w.freq.dt * s)
        fa = g3.aca3_compress(ctx, T, F, "slp", eps3=1e-4, dense_face_max=-1, residual_face_max=residual_face_max)
        y = g3.apply_gcq(ctx, T, None, fa, W)
        out.append((fa.stats(), fa.ranks(), y.cpu().numpy() / s))
    (s0, r0, y0), (s1, r1, y1) = out
    assert (s0["entries_face_dense"] > 0) == (residual_face_max == 0)
    assert s0["entries"] == s1["entries"] and s0["face_rank_sum"] == s1["face_rank_sum"]
    assert np.array_equal(r0, r1)
    assert np.linalg.norm(y1 - y0) <= 2e-6 * np.linalg.norm(y0)   # float32 sums in another order
