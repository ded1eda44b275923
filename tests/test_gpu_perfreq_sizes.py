"""The per-frequency apply at the edges of its far-field kernels' tiles.

Every column against the float64 dense oracle on sampled rows: the compression
bounds a block's error over all Ku unique frequencies together by eps3 = 1e-4 of
its norm over them, so one frequency's by sqrt(Ku) eps3.  And the columns'
sum against the sum over the frequencies, which other kernels form from the
same factors (float64: 1e-12, float32: 1e-5).  The sizes: one and several
chunks of right-hand sides and of frequencies (K = 2, 30, 34, 130: 2, 16, 18
and 66 unique), low-rank blocks of more than 64 rows and columns and of a
few, dense-face blocks of more than 32 rows and of odd sizes.
"""
import numpy as np
import pytest

from inputs import meshes
from oracle import apply as O_apply, freqs as O_freqs, quadrature as O_q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf,K,dense,prec", [
    (5, 32, 2, 0, "mixed"), (5, 9, 30, -1, "mixed"), (6, 51, 34, 90 * 90, "mixed"), (9, 32, 34, -1, "mixed"),
    (7, 32, 130, 0, "mixed"), (9, 40, 34, -1, "fp64"), (5, 47, 130, 90 * 90, "fp64")])
def test_perfreq_sizes(g3, n, leaf, K, dense, prec):
    import torch
    ctx = g3.Context(0)
    v, t = meshes.cube(n)
    E = t.shape[0]
    s = O_freqs.bdf2(K, 0.7 * 1.1 / n, 1e-8 ** (1 / (2 * K)))
    T = g3.build_cluster_tree(ctx, v, t, leaf, 1.0)
    F = g3.g3_freqs_from_array(ctx, s)
    W = np.random.default_rng(K).standard_normal((E, K, 2)) @ np.array([1.0, 1j])
    Wd = torch.from_numpy(W).to("cuda", torch.complex64 if prec == "mixed" else torch.complex128)
    nf = g3.assemble_near(ctx, T, F, "slp", prec=prec)
    fa = g3.aca3_compress(ctx, T, F, "slp", prec=prec, eps3=1e-4, dense_face_max=dense)
    Y = g3.apply_gcq(ctx, T, nf, fa, Wd, mode="perfreq").cpu().numpy()
    y = g3.apply_gcq(ctx, T, nf, fa, Wd).cpu().numpy()
    assert np.linalg.norm(Y.sum(axis=1) - y) <= (1e-12 if prec == "fp64" else 1e-5) * np.linalg.norm(y)
    geo = O_q.Geometry(v, t)
    rows = np.arange(0, E, max(1, E // 24))
    Yref = O_apply.dense_apply_perfreq(lambda I, J, z: O_q.entries(geo, "slp", I, J, z), E, s, W, rows=rows)
    err = np.linalg.norm(Y[rows] - Yref, axis=0) / np.linalg.norm(Yref, axis=0)
    assert err.max() <= 1e-4 * np.sqrt(F.info()[1]), err
