"""Regular near-field entries (power series in the frequency, point by point beyond)
against the point-by-point float64 entries of g3_entries."""
from __future__ import annotations

import numpy as np
import pytest

from inputs import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,scheme", [("slp", "colloc7"), ("dlp", "colloc7"), ("slp", "galerkin4x4")])
@pytest.mark.parametrize("shape,n,leaf", [("cube", 3, 7), ("sphere", 1, 32)])
def test_regular_entries_all_degrees(g3, kernel, scheme, shape, n, leaf):
    v, t = meshes.cube(n) if shape == "cube" else meshes.icosphere(n)
    v = v * np.array([1.0, 0.3, 1.7])   # unequal triangles: one frequency meets several degrees in a warp
    h = float(np.linalg.norm(v[t[:, 1]] - v[t[:, 0]], axis=1).max())
    D = float(np.linalg.norm(v.max(axis=0) - v.min(axis=0)))
    # |s| h from almost 0 through each degree's limit to point by point; 49 frequencies: three chunks
    z = np.concatenate([[1e-9, 1e-6], np.geomspace(0.05, 40.0, 47)]) / h
    s = z * np.exp(1j * np.linspace(0.0, 1.5, z.size))
    ctx = g3.Context(0)
    T = g3.build_cluster_tree(ctx, v, t, leaf, 1.0)
    F = g3.g3_freqs_from_array(ctx, s)
    R = g3.g3_freqs_from_array(ctx, s.real.copy())
    Ku, info, ks = F.info()[1], T.get(), np.arange(z.size)
    tv = t[info["perm"]]
    sr = np.abs(s) * D
    # float64: the reference rounds its phases; float32: frequency, distance and phase
    # rounded (4 |s| r), the sine and cosine, and 17 terms of at most exp(2.25)
    for prec, tol in (("fp64", 2.0 ** -52 * (2 * sr + 24 * np.exp(2.0))), ("mixed", 2.0 ** -24 * (4 * sr + 150))):
        nf = g3.assemble_near(ctx, T, F, kernel, scheme=scheme, prec=prec)
        seen = 0
        for b, (rb, re, cb, ce, far) in enumerate(info["blocks"]):
            if far:
                continue
            I, J = (x.ravel() for x in np.meshgrid(np.arange(rb, re), np.arange(cb, ce), indexing="ij"))
            if scheme == "galerkin4x4":   # (pairs with a common vertex have their own rule)
                ok = ~(tv[I][:, :, None] == tv[J][:, None, :]).any(axis=(1, 2))
            else:
                ok = I != J
            if not ok.any():
                continue
            A = nf.block(b, re - rb, ce - cb, Ku)[:, (I - rb)[ok], (J - cb)[ok]].T
            ids = info["perm"][I[ok]], info["perm"][J[ok]]
            ref = g3.g3_entries(ctx, T, F, kernel, *ids, ks, "fp64", scheme)
            # the sum of the terms' absolute values: the entry at the real part (double layer:
            # times 1 + |s| r for its factor 1 + s r)
            mag = np.abs(g3.g3_entries(ctx, T, R, kernel, *ids, ks, "fp64", scheme))
            if kernel == "dlp":
                mag = mag * (1 + sr)
            # (double layer: the distance from the plane is rounded against the distance)
            lim = tol * mag + (8 * tol[0] / 150 * mag.max(axis=0) if kernel == "dlp" else 0) + 1e-36
            assert (np.abs(A - ref) <= lim).all(), (prec, b, float((np.abs(A - ref) / lim).max()))
            seen += int(ok.sum())
        assert seen > 0
