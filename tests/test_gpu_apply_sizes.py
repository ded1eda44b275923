"""The sum over the frequencies against the per-frequency apply (other kernels) summed on the
host: leaf sizes at the edges of the near field's stages and lanes, odd slabs, both precisions,
dense and low-rank far fields, with and without the tensor cores."""
from __future__ import annotations

import numpy as np
import pytest

from inputs import meshes

pytestmark = pytest.mark.gpu


# rows per leaf cluster: 6, odd ones (slabs that start at odd elements), 32 | 33 (one or two
# rows per lane), 96 (pieces of a few columns), 768 (one leaf, beyond a stage: the wide kernel)
@pytest.mark.parametrize("leaf", [7, 15, 32, 40, 96, 768])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_sum_against_per_frequency(leaf, prec):
    import torch

    import paper_2312_11219_gb300 as g3
    v, t = meshes.cube(8) if leaf != 15 else meshes.cube(7)      # 768, or 588 triangles (leaves of 9 and 10)
    dt = torch.complex64 if prec == "mixed" else torch.complex128
    tol = 5e-6 if prec == "mixed" else 1e-12   # float32 sums of up to 1e5 terms: ~3e-7 sqrt-like growth, x 15
    ctx = g3.Context(0)
    T = g3.build_cluster_tree(ctx, v, t, leaf, 1.0)
    F = g3.g3_freqs_bdf2(ctx, 22, 1e-8 ** (1 / 44), 0.1)          # 12 unique frequencies
    near = g3.assemble_near(ctx, T, F, "slp", prec=prec)
    M = T.info()["ne"]
    gen = torch.Generator("cuda").manual_seed(3)
    W = torch.randn(22, M, dtype=dt, device="cuda", generator=gen).t()
    fars = [None]
    if T.info()["n_far"]:
        fars += [g3.aca3_compress(ctx, T, F, "slp", prec=prec, eps3=1e-4, dense_face_max=d) for d in (0, -1)]
    for far in fars:
        ref = g3.apply_gcq(ctx, T, near, far, W, mode="perfreq").sum(1).cpu().numpy()
        for tc in (True, False):
            ctx.set_apply_tensor_cores(tc)
            y = g3.apply_gcq(ctx, T, near, far, W).cpu().numpy()
            assert np.linalg.norm(y - ref) <= tol * np.linalg.norm(ref), (leaf, prec, far is None, tc)
        ctx.set_apply_tensor_cores(True)
