"""Every set-up and apply on a non-blocking stream, with the legacy stream busy.

The library's copies and clears must be ordered on the context's own stream: a
torch stream has no ordering with the legacy one, on which 30 ms of products are
queued before each call, so that anything left there would come too late.  The
results are those of a context on the idle legacy stream (float32 sums to 2e-6,
ranks and frequencies equal).
"""
import numpy as np
import pytest

from inputs import workloads

pytestmark = pytest.mark.gpu


def _chain(g3, ctx, torch, before):
    """{name: array} of every call; before() runs ahead of each."""
    def call(f, *a, **k):
        before()
        return f(*a, **k)

    def dev(W):
        t = torch.empty(W.T.shape, dtype=torch.complex64, device="cuda")
        t.copy_(torch.from_numpy(np.ascontiguousarray(W.T)).to(torch.complex64))
        torch.cuda.current_stream().synchronize()
        return t.t()

    out = {}
    w = workloads.get("cube768")
    W = dev(workloads.densities(w.E, w.freq.K, 3))
    T = call(g3.build_cluster_tree, ctx, w.verts, w.tris, w.leaf, w.eta)
    F = call(g3.freqs_from_spec, ctx, w.freq)
    Fa = call(g3.g3_freqs_from_array, ctx, F.get()["s"])
    out["entries"] = call(g3.g3_entries, ctx, T, Fa, "slp", [0, 5, 9], [700, 3, 9], [0, 7, 20])
    nf = call(g3.assemble_near, ctx, T, F, "slp")
    for name, d in (("dense", 48 * 48), ("low", -1)):
        fa = call(g3.aca3_compress, ctx, T, F, "slp", eps3=1e-4, dense_face_max=d)
        out["ranks " + name] = fa.ranks()
        out["y " + name] = call(g3.apply_gcq, ctx, T, nf, fa, W)
        out["perfreq " + name] = call(g3.apply_gcq, ctx, T, nf, fa, W, mode="perfreq")
    spill = call(g3.aca3_compress, ctx, T, F, "slp", eps3=1e-4, dense_face_max=-1, pool_factor=0.02)
    assert spill.stats()["spilled_blocks"] > 0
    out["ranks spilled"] = spill.ranks()
    out["labels"] = call(fa.labels)
    X = call(g3.block_features, ctx, T, F, "slp", 1e-4)
    net = call(g3.mlp_train, ctx, X, out["labels"], epochs=3, batch=64, seed=3)
    out["predicted"] = call(net.predict, X)
    out["ranks k1"] = call(g3.aca3_compress, ctx, T, F, "slp", eps3=1e-4, k1=np.zeros(len(X), np.int32)).ranks()
    # the H-matrix as a whole, with a factor pool that grows
    fw = call(g3.aca3_compress, ctx, T, F, "slp", eps3=1e-6, whole_matrix=1, face_rank_max=8)
    b = T.get()["blocks"]
    b = b[b[:, 4] == 1]
    m, n = b[:, 1] - b[:, 0], b[:, 3] - b[:, 2]
    assert fw.stats()["factor_bytes"] > 8 * 4 * int((8 * (m + n) + F.info()[1]).sum())
    out["ranks whole"] = fw.ranks()
    out["y whole"] = call(g3.apply_gcq, ctx, T, None, fw, W)
    # two meshes in one launch
    w2 = workloads.get("cube192")
    T2 = call(g3.build_cluster_tree, ctx, w2.verts, w2.tris, 8, w2.eta)
    F2 = call(g3.g3_freqs_gcq, ctx, 16, 0.005, 0.015)
    fas = call(g3.aca3_compress_batch, ctx, [T, T2], [F, F2], "dlp", eps3=1e-4)
    n2 = call(g3.assemble_near, ctx, T2, F2, "dlp")
    out["y batch"] = call(g3.apply_gcq, ctx, T, None, fas[0], W)
    out["y batch 2"] = call(g3.apply_gcq, ctx, T2, n2, fas[1], dev(workloads.densities(w2.E, 16, 4)))
    # Galerkin: constant and linear elements
    ws = workloads.get("sphere320g")
    Ts = call(g3.build_cluster_tree, ctx, ws.verts, ws.tris, ws.leaf, ws.eta)
    Fs = call(g3.g3_freqs_gcq, ctx, 16, 0.005, 0.015)
    ng = call(g3.assemble_near, ctx, Ts, Fs, "slp", "galerkin4x4")
    fg = call(g3.aca3_compress, ctx, Ts, Fs, "slp", "galerkin4x4", eps3=1e-4)
    out["y galerkin"] = call(g3.apply_gcq, ctx, Ts, ng, fg, dev(workloads.densities(ws.E, 16, 5)))
    Tp = call(g3.build_p1_tree, ctx, Ts)
    nh = call(g3.assemble_near, ctx, Tp, Fs, "hyp", "galerkin4x4")
    fh = call(g3.aca3_compress, ctx, Tp, Fs, "hyp", "galerkin4x4", eps3=1e-4)
    out["y hyp"] = call(g3.apply_gcq, ctx, Tp, nh, fh, dev(workloads.densities(ws.verts.shape[0], 16, 6)))
    a, bb, c = (np.random.default_rng(7).standard_normal((3, k)) + 0j for k in (60, 50, 12))
    out["separable"] = call(g3.aca3_compress_separable, ctx, a, bb, c, prec="mixed", eps3=1e-4).ranks()
    return {k: v.cpu().numpy() if hasattr(v, "cpu") else np.asarray(v) for k, v in out.items()}


def test_non_blocking_stream_with_the_legacy_stream_busy(g3):
    import torch
    ref = _chain(g3, g3.Context(0), torch, lambda: None)
    x = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    side, legacy = torch.cuda.Stream(), torch.cuda.default_stream()

    def busy():
        nonlocal x
        with torch.cuda.stream(legacy):
            for _ in range(12):
                x = (x @ x).clamp_(-1, 1)

    with torch.cuda.stream(side):
        got = _chain(g3, g3.Context(0, side.cuda_stream), torch, busy)
    torch.cuda.synchronize()
    for k, r in ref.items():
        if r.dtype.kind == "i":
            assert np.array_equal(got[k], r), k
        else:
            assert np.linalg.norm(got[k] - r) <= 2e-6 * np.linalg.norm(r), k
