"""Single-layer self entries of the near field (moment series about 0 and about the
middle radius, direct sum) against the point-by-point float64 routine of g3_entries."""
from __future__ import annotations

import numpy as np
import pytest

from inputs import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n", [("cube", 3), ("sphere", 1)])
def test_self_entries_all_branches(shape, n):
    import paper_2312_11219_gb300 as g3
    v, t = meshes.cube(n) if shape == "cube" else meshes.icosphere(n)
    v = v * np.array([1.0, 0.3, 1.7])   # unequal triangles: one frequency meets several branches
    h = float(np.linalg.norm(v[t[:, 1]] - v[t[:, 0]], axis=1).max())
    # |s| h from almost 0 through each branch's edge (|s| rmax = 4, |s| rh = 4) to far beyond; 37
    # frequencies: more than one per lane
    z = np.concatenate([[1e-9, 1e-6], np.geomspace(0.05, 150.0, 35)]) / h
    s = z * np.exp(1j * np.linspace(0.0, 1.5, z.size))
    ctx = g3.Context(0)
    T = g3.build_cluster_tree(ctx, v, t, 8, 1.0)
    F = g3.g3_freqs_from_array(ctx, s)
    Ku = F.info()[1]
    info = T.get()
    E = T.info()["ne"]
    ids = np.arange(E)
    ref = g3.g3_entries(ctx, T, F, "slp", ids, ids, np.arange(z.size), "fp64")
    for prec, tol in (("fp64", 1e-12), ("mixed", 1.2e-7)):   # series: e^4 x 2^-53 and less; float32: one rounding
        nf = g3.assemble_near(ctx, T, F, "slp", prec=prec)
        seen = 0
        for b, (rb, re, cb, ce, far) in enumerate(info["blocks"]):
            if far or rb != cb:
                continue
            A = nf.block(b, re - rb, ce - cb, Ku)
            d = np.einsum("kii->ik", A)
            want = ref[info["perm"][rb:re]]
            err = np.abs(d - want) / np.abs(want)
            assert err.max() <= tol, (prec, float(err.max()))
            seen += re - rb
        assert seen == E
