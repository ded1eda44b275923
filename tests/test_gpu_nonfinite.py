"""A density that is not finite stays visible in the far field.

One value of W is set to the NaN that GPU arithmetic produces (0x7fffffff, whose
rounding to TF32 wraps to -0 when it is done on the bits alone), to the quiet NaN
of the host or to an infinity.  The far field alone and the whole sum, with dense
and with low-rank faces, must then be non-finite on the same rows with the x
formation on the tensor cores and on the CUDA cores, and agree on the others to the
bound of the two orders of float32 sums (2e-6).
"""
import numpy as np
import pytest

from inputs import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ops(g3):
    ctx = g3.Context(0)
    w = workloads.get("cube768")
    T = g3.build_cluster_tree(ctx, w.verts, w.tris, w.leaf, w.eta)
    F = g3.freqs_from_spec(ctx, w.freq)
    nf = g3.assemble_near(ctx, T, F, "slp")
    fas = {d: g3.aca3_compress(ctx, T, F, "slp", eps3=w.eps3, dense_face_max=d) for d in (48 * 48, -1)}
    assert fas[48 * 48].stats()["dense_crosses"] > 0 and fas[-1].stats()["dense_crosses"] == 0
    return ctx, w, T, nf, fas


@pytest.mark.parametrize("bits", [0x7FFFFFFF, 0x7FC00000, -0x400000, 0x7F800000, -0x800000])
@pytest.mark.parametrize("dense", [48 * 48, -1])
def test_non_finite_density(g3, ops, dense, bits):
    import torch
    ctx, w, T, nf, fas = ops
    W = torch.from_numpy(workloads.densities(w.E, w.freq.K, 3).T.copy()).to("cuda", torch.complex64)
    torch.view_as_real(W).view(torch.int32)[5, 100, 0] = bits
    W = W.t()
    out = {}
    for tc in (True, False):
        ctx.set_apply_tensor_cores(tc)
        Y = torch.empty(w.E, dtype=torch.complex64, device="cuda")
        g3.apply_gcq_noalloc(ctx, T, nf, fas[dense], W, Y)
        out[tc] = [g3.apply_gcq(ctx, T, None, fas[dense], W).cpu().numpy(),
                   g3.apply_gcq(ctx, T, nf, fas[dense], W).cpu().numpy(), Y.cpu().numpy()]
    ctx.set_apply_tensor_cores(True)
    for a, b in zip(out[True], out[False]):
        ok = np.isfinite(b)
        assert not ok.all()
        assert np.array_equal(np.isfinite(a), ok)
        assert np.linalg.norm(a[ok] - b[ok]) <= 2e-6 * max(np.linalg.norm(b[ok]), 1e-300)
    assert np.isfinite(out[False][0]).any()   # rows without a far block to the element
