"""What a program does with this library, as cases that can be timed.

A boundary element program with (generalised) convolution quadrature sets an
operator up once (cluster tree, frequencies, near field, three-way ACA) and
then applies it to the densities of every time step.  The cases are those two
halves, alone and together, over the meshes, operators, frequency sets and
precisions of this repository's workloads:

  step      mesh on the host -> tree, frequencies, near field, compression and
            one apply: the whole call chain of a small problem;
  setup     near field, compression and the first apply on a tree in hand;
  near      near field and its product alone;
  batch     several meshes compressed in one launch, each with its apply;
  apply     one apply of an operator in hand: the sum over the frequencies,
            the per-frequency form, or the allocation-free form;
  march     time steps of the gCQ solver: history update and apply per step.

Densities have the precision of the operator: complex64 with mixed precision,
complex128 with float64.  The seed moves and scales the mesh by a little (the
time step stays) and draws the densities.
"""
import functools
import math

import numpy as np
import torch

import paper_2312_11219_gb300 as g3
from inputs import meshes

DEV = "cuda:0"
DT_MIN, DT_MAX = 0.005, 0.015      # graded steps of the gCQ sets
EPS3 = 1e-4
LEAF, ETA = 32, 1.0


def _case(name, do, shape, n, kernel, K, freqs="bdf2", scheme="colloc7", prec="mixed", max_block=0, mode="sum",
          host=False, meshes=1):
    return {"name": name, "do": do, "shape": shape, "n": n, "kernel": kernel, "K": K, "freqs": freqs,
            "scheme": scheme, "prec": prec, "max_block": max_block, "mode": mode, "host": host, "meshes": meshes}


def listed():
    return [
        # the smallest problem in use, from host arrays to host arrays: a unit
        # cube of 768 triangles; launches, allocations and latency count
        _case("step-cube768", "step", "cube", 8, "slp", 32, host=True),
        # a float64 operator (the accuracy reference a user checks against)
        _case("step-lshape768-fp64", "step", "lshape", 8, "dlp", 32, prec="fp64"),
        # a middle-sized operator on the plain partition, double layer
        _case("setup-lshape3072-dlp", "setup", "lshape", 16, "dlp", 64),
        # the headline problem: the 12,288-triangle L-shape, single layer
        _case("setup-lshape12288-slp", "setup", "lshape", 32, "slp", 128, max_block=192),
        # Galerkin single layer on the sphere, gCQ frequencies
        _case("setup-sphere5120-galerkin", "setup", "sphere", 4, "slp", 64, "gcq", "galerkin4x4", max_block=192),
        # the Neumann problem: hypersingular operator, linear elements
        _case("setup-sphere1280-hyp", "setup", "sphere", 3, "hyp", 64, "gcq", "galerkin4x4"),
        # near-field assembly of the headline problem (ragged blocks, self terms)
        _case("near-lshape12288-slp", "near", "lshape", 32, "slp", 128, max_block=192),
        # several bodies compressed in one launch (odd sizes, one K for each)
        _case("batch-6-slp", "batch", "mixed", 13, "slp", 64, max_block=192, meshes=6),
        # the apply of every time step on the headline problem, double layer
        _case("apply-lshape12288-dlp", "apply", "lshape", 32, "dlp", 128, max_block=192),
        # the allocation-free apply of a small operator: launch latency
        _case("apply-noalloc-cube1728", "apply", "cube", 12, "slp", 32, mode="noalloc"),
        # A(s_l) w_l for every frequency by itself
        _case("apply-perfreq-lshape3072", "apply", "lshape", 16, "slp", 64, mode="perfreq"),
        # four time steps of the gCQ solver on a 20,480-triangle sphere: W and
        # the history (42 MB each) move through every step
        _case("march-sphere20480", "march", "sphere", 5, "slp", 256, "gcq", max_block=192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["step", "step", "setup", "setup", "setup", "near", "batch", "apply", "apply", "apply", "march"])
    shape = "sphere" if do == "march" else rng.choice(["cube", "cube", "lshape", "sphere"])
    if do == "batch":
        return {k: v for k, v in _case("", do, "mixed", _log_int(rng, 7, 15), rng.choice(["slp", "dlp"]),
                                       2 * _log_int(rng, 16, 32), max_block=192,
                                       meshes=rng.randint(2, 6)).items() if k != "name"}
    hi = {"step": 11, "setup": 22, "near": 30, "apply": 28}.get(do, 28)   # squares per cube edge
    n = (_log_int(rng, 4, hi) if shape == "cube" else 2 * _log_int(rng, 3, hi // 2) if shape == "lshape"
         else rng.randint(2, 3 if do == "step" else 4))
    E = 20 * 4 ** n if shape == "sphere" else 12 * n * n
    kernel, scheme, prec, mode = rng.choice(["slp", "dlp"]), "colloc7", "mixed", "sum"
    freqs = "gcq" if shape == "sphere" and (do == "march" or rng.random() < 0.5) else "bdf2"
    K = 2 * _log_int(rng, 8, 64 if E <= 6144 else 48)
    if do == "setup" and shape == "sphere" and rng.random() < 0.5:
        scheme, freqs, kernel = "galerkin4x4", "gcq", "hyp" if n < 4 and rng.random() < 0.4 else "slp"
        K = min(K, 64)
    elif do == "step" and E <= 768 and rng.random() < 0.4:
        prec, K = "fp64", min(K, 32)
    elif do == "apply":
        mode = rng.choice(["sum", "sum", "perfreq", "noalloc"])
        if mode == "perfreq":
            K = min(K, 64)
    max_block = 192 if E > 3072 else rng.choice([0, 192])
    host = do == "step" and rng.random() < 0.5
    c = _case("", do, shape, n, kernel, K, freqs, scheme, prec, max_block, mode, host)
    c.pop("name")
    return c


# ---- inputs ------------------------------------------------------------------------------

@functools.lru_cache(maxsize=32)
def _base(shape, n):
    if shape == "cube":
        return meshes.cube(n)
    if shape == "lshape":
        return meshes.lshape(n)
    return meshes.icosphere(n)


def _shapes(case):
    """(shape, n) of every mesh: one, or the batch's cubes of growing odd sizes and spheres."""
    if case["do"] != "batch":
        return [(case["shape"], case["n"])]
    return [("sphere", 3) if g % 3 == 2 else ("cube", case["n"] + 2 * (g % 3) - g // 3) for g in range(case["meshes"])]


def _mesh(shape, n, rng):
    v, t = _base(shape, n)
    return np.ascontiguousarray(v * rng.uniform(0.95, 1.05) + rng.uniform(-1.0, 1.0, 3)), t


def _inputs(case, seed):
    """The meshes [(verts, tris)] and the densities [W (rows, K), columns contiguous] of a case."""
    rng = np.random.default_rng(seed)
    ms = [_mesh(s, n, rng) for s, n in _shapes(case)]
    gen = torch.Generator(DEV).manual_seed(int(seed))
    dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    rows = [v.shape[0] if case["kernel"] in ("hyp", "adj") else t.shape[0] for v, t in ms]
    return ms, [torch.randn(case["K"], m, dtype=dt, device=DEV, generator=gen).t() for m in rows]


def _dt(case, g=0):
    """Step of the multistep frequencies: 0.7 mean edge lengths of the unscaled mesh."""
    v, t = _base(*_shapes(case)[g])
    return 0.7 * float(np.linalg.norm(v[t[:, 1]] - v[t[:, 0]], axis=1).mean())


def _lam(K):
    return 1e-8 ** (1.0 / (2 * K))


def _freqs(ctx, case, g=0):
    if case["freqs"] == "gcq":
        return g3.g3_freqs_gcq(ctx, case["K"], DT_MIN, DT_MAX)
    return g3.g3_freqs_bdf2(ctx, case["K"], _lam(case["K"]), _dt(case, g))


def _tree(ctx, case, v, t):
    T = g3.build_cluster_tree(ctx, v, t, LEAF, ETA, max_block=case["max_block"])
    return g3.build_p1_tree(ctx, T) if case["kernel"] in ("hyp", "adj") else T


def prepare(case, seed):
    ms, Ws = _inputs(case, seed)
    ctx = g3.Context(0)
    st = {"case": case, "ctx": ctx, "meshes": ms, "W": Ws}
    if case["do"] == "step":
        if case["host"]:
            st["W"] = [np.asfortranarray(W.cpu().numpy()) for W in Ws]
        return st
    st["T"] = [_tree(ctx, case, v, t) for v, t in ms]
    st["F"] = [_freqs(ctx, case, g) for g in range(len(ms))]
    if case["do"] in ("apply", "march"):
        T, F, a = st["T"][0], st["F"][0], (case["kernel"], case["scheme"], case["prec"])
        st["near"] = g3.assemble_near(ctx, T, F, *a)
        st["fac"] = g3.aca3_compress(ctx, T, F, *a, eps3=EPS3)
    if case["do"] == "apply" and case["mode"] == "noalloc":
        st["Y"] = torch.empty(Ws[0].shape[0], dtype=Ws[0].dtype, device=DEV)
    if case["do"] == "march":
        st["theta"] = [W[:, n].contiguous() for W in Ws for n in range(STEPS)]
        st["X"] = torch.zeros_like(Ws[0].t()).t()
        st["Wn"] = torch.empty_like(Ws[0].t()).t()
    return st


STEPS = 4
DTS = [0.01 * (1.0 + 0.5 * math.sin(2.0 * math.pi * n / 64.0)) for n in range(1, STEPS + 2)]


# ---- one pass ------------------------------------------------------------------------------

def run(st):
    case, ctx = st["case"], st["ctx"]
    a = (case["kernel"], case["scheme"], case["prec"])
    do = case["do"]
    if do == "step":
        (v, t), W = st["meshes"][0], st["W"][0]
        T = _tree(ctx, case, v, t)
        F = _freqs(ctx, case)
        near = g3.assemble_near(ctx, T, F, *a)
        fac = g3.aca3_compress(ctx, T, F, *a, eps3=EPS3)
        return g3.apply_gcq(ctx, T, near, fac, W)
    if do == "setup":
        T, F = st["T"][0], st["F"][0]
        near = g3.assemble_near(ctx, T, F, *a)
        fac = g3.aca3_compress(ctx, T, F, *a, eps3=EPS3)
        return g3.apply_gcq(ctx, T, near, fac, st["W"][0])
    if do == "near":
        T = st["T"][0]
        near = g3.assemble_near(ctx, T, st["F"][0], *a)
        return g3.apply_gcq(ctx, T, near, None, st["W"][0])
    if do == "batch":
        fas = g3.aca3_compress_batch(ctx, st["T"], st["F"], *a, eps3=EPS3)
        return [g3.apply_gcq(ctx, T, g3.assemble_near(ctx, T, F, *a), fa, W)
                for T, F, fa, W in zip(st["T"], st["F"], fas, st["W"])]
    if do == "apply":
        if case["mode"] == "noalloc":
            return g3.apply_gcq_noalloc(ctx, st["T"][0], st["near"], st["fac"], st["W"][0], st["Y"])
        return g3.apply_gcq(ctx, st["T"][0], st["near"], st["fac"], st["W"][0], mode=case["mode"])
    st["X"].zero_()
    ys = []
    for n in range(STEPS):
        Wn = g3.gcq_history(ctx, st["F"][0], st["X"], st["theta"][n], DTS[n], DTS[n + 1], W=st["Wn"])
        ys.append(g3.apply_gcq(ctx, st["T"][0], st["near"], st["fac"], Wn))
    return {"y": ys, "X": st["X"]}


# ---- the work a pass cannot do without -------------------------------------------------------

def _partition(v, t, max_block):
    """perm and the blocks [(rows, columns, admissible)] of the balanced cluster tree: longest box
    side, left half of the order by (centroid, index), leaves of at most LEAF; a pair is admissible
    when min(diam)^2 <= ETA^2 dist^2 > 0 (capped: and no side above max_block that can be split)."""
    c = ((v[t[:, 0]] + v[t[:, 1]]) + v[t[:, 2]]) / 3.0
    lo_e, hi_e = v[t].min(axis=1), v[t].max(axis=1)
    perm = np.arange(t.shape[0])
    nodes = []   # begin, end, left, right, lo, hi, diam^2

    def build(b, e):
        i = len(nodes)
        idx = perm[b:e]
        lo, hi = lo_e[idx].min(axis=0), hi_e[idx].max(axis=0)
        ext = hi - lo
        nodes.append([b, e, -1, -1, lo.tolist(), hi.tolist(), float((ext[0] * ext[0] + ext[1] * ext[1]) + ext[2] * ext[2])])
        if e - b > LEAF:
            ax = int(np.argmax(ext))
            perm[b:e] = idx[np.lexsort((idx, c[idx, ax]))]
            m = b + (e - b) // 2
            nodes[i][2], nodes[i][3] = build(b, m), build(m, e)
        return i

    build(0, t.shape[0])
    out, stack = [], [(0, 0)]
    while stack:
        i, j = stack.pop()
        a, b = nodes[i], nodes[j]
        d2 = 0.0
        for k in range(3):
            g = max(a[4][k] - b[5][k], b[4][k] - a[5][k], 0.0)
            d2 += g * g
        adm = d2 > 0.0 and min(a[6], b[6]) <= ETA * ETA * d2
        la, lb = a[2] < 0, b[2] < 0
        if adm and (not max_block or max(a[1] - a[0], b[1] - b[0]) <= max_block or (la and lb)):
            out.append((a[0], a[1], b[0], b[1], True))
        elif la and lb:
            out.append((a[0], a[1], b[0], b[1], False))
        else:
            stack += [(x, y) for x in ([i] if la else a[2:4]) for y in ([j] if lb else b[2:4])]
    return perm, out


@functools.lru_cache(maxsize=64)
def _counts(shape, n, max_block):
    """Near-field entries per frequency and (rows, columns) sums over the far blocks."""
    _, blocks = _partition(*_base(shape, n), max_block)
    near = sum((b - a) * (d - c) for a, b, c, d, f in blocks if not f)
    far = [(b - a, d - c) for a, b, c, d, f in blocks if f]
    return near, sum(m + k for m, k in far), len(far), shape and _base(shape, n)[1].shape[0], sum(m * k for m, k in far)


#: Crosses of a block and face ranks that a tolerance of 1e-4 takes, at the least (the means over the workloads' blocks are
#: above them), and floating operations of one entry: 7 points or 16 pairs of points, each an exponential, a sine, a cosine, a
#: root and some ten multiply-adds.
CROSSES, RANK, OPS = 6, 7, {"colloc7": 7 * 24, "galerkin4x4": 16 * 24}


def work(case):
    s = 16 if case["prec"] == "fp64" else 8
    K, Ku = case["K"], case["K"] // 2 + (case["freqs"] == "bdf2")
    B = Fl = 0.0
    for shape, n in _shapes(case):
        near, mn, nb, E, pairs = _counts(shape, n, case["max_block"])
        p = 9 if case["kernel"] in ("hyp", "adj") else 1
        rows = _base(shape, n)[0].shape[0] if p == 9 else E
        lines = CROSSES * RANK * mn * (3 if p == 9 else 1)    # values of all faces' rows and columns
        fac = min(lines + CROSSES * nb * Ku, p * pairs * Ku)  # stored factor values
        ops = OPS[case["scheme"]]
        if case["do"] in ("apply", "march"):
            m = STEPS if case["do"] == "march" else 1
            out = K if case["mode"] == "perfreq" else 1
            B += m * s * (p * near * Ku + fac + rows * (K + out))
            Fl += m * 16.0 * (p * near * Ku + fac * (Ku if case["mode"] == "perfreq" else 1))
            if case["do"] == "march":
                B += m * 3.0 * s * rows * K
        else:
            far = case["do"] != "near"
            # geometry and densities in, near field and factors written and read once, y out
            B += 53 * 4.0 * E + s * rows * (K + 1) + 2.0 * s * (p * near * Ku + far * fac)
            Fl += (ops + 16.0) * (p * near * Ku + far * (lines + CROSSES * nb * Ku))
    return {"bytes": B, "flops": Fl}


# ---- what a pass returns, in 64 bits ---------------------------------------------------------

def _jacobi(u, m):
    """sn, cn, dn of real u (descending Landen transformation) and K(m)."""
    a, b, c = [1.0], math.sqrt(1.0 - m), [math.sqrt(m)]
    while abs(c[-1]) > 1e-16 and len(a) < 20:
        a, c, b = a + [0.5 * (a[-1] + b)], c + [0.5 * (a[-1] - b)], math.sqrt(a[-1] * b)
    N = len(a) - 1
    ph = 2.0 ** N * a[N] * u
    prev = ph
    for n in range(N, 0, -1):
        prev, ph = ph, 0.5 * (ph + np.arcsin(c[n] * np.sin(ph) / a[n]))
    return np.sin(ph), np.cos(ph), np.cos(ph) / np.cos(prev - ph), math.pi / (2.0 * a[N])


def _s(case, g=0):
    """All frequencies s_l, the contour weights (gCQ) and the unique half with its partners."""
    K = case["K"]
    if case["freqs"] == "bdf2":
        z = 1.0 - _lam(K) * np.exp(2j * np.pi * np.arange(K) / K)
        return (z + 0.5 * z * z) / _dt(case, g), None, np.arange(K // 2 + 1), (K - np.arange(K)) % K
    q = DT_MAX / DT_MIN
    r = math.sqrt(2.0 * q - 1.0)
    k = (q - r) / (q + r)
    m = k * k
    Kk, Kp = _jacobi(0.0, m)[3], _jacobi(0.0, 1.0 - m)[3]
    s, c, d, _ = _jacobi(-Kk + (np.arange(1, K + 1) - 0.5) * 4.0 * Kk / K, m)
    s1, c1, d1, _ = _jacobi(np.float64(0.5 * Kp), 1.0 - m)
    den = c1 * c1 + m * s * s * s1 * s1
    sn = (s * d1 + 1j * c * d * s1 * c1) / den
    cn = (c * c1 - 1j * s * d * s1 * d1) / den
    dn = (d * c1 * d1 - 1j * m * s * c * s1) / den
    pref = 1.0 / (DT_MIN * (q - 1.0))
    ss = pref * (r * (1.0 / k + sn) / (1.0 / k - sn) - 1.0)
    om = -4.0 * Kk * pref * r * 2.0 * cn * dn / (k * (1.0 / k - sn) ** 2) / (2j * np.pi * K)
    return ss, om, np.arange(K // 2), K - 1 - np.arange(K)


def _f64(x):
    return torch.as_tensor(np.ascontiguousarray(x), device=DEV)


def _panels(v, t):
    P = _f64(v)[_f64(t).long()]                                  # [E, 3 vertices, 3]
    n = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    a2 = n.norm(dim=1, keepdim=True)
    return P, n / a2, 0.5 * a2[:, 0]


def _radon7():
    r = math.sqrt(15.0)
    a1, b1, a2, b2 = (6 - r) / 21, (9 + 2 * r) / 21, (6 + r) / 21, (9 - 2 * r) / 21
    L = [[1 / 3] * 3, [a1, a1, b1], [a1, b1, a1], [b1, a1, a1], [a2, a2, b2], [a2, b2, a2], [b2, a2, a2]]
    return _f64(L), _f64([9 / 40] + [(155 - r) / 1200] * 3 + [(155 + r) / 1200] * 3)


def _conical4():
    r = math.sqrt(6.0)
    pts, w = [], []
    for u, wu in (((4 - r) / 10, (9 + r) / 36), ((4 + r) / 10, (9 - r) / 36)):
        for x in (0.5 - 0.5 / math.sqrt(3), 0.5 + 0.5 / math.sqrt(3)):
            l2 = x * (1 - u)
            pts.append([1 - u - l2, u, l2])
            w.append(wu)
    return _f64(pts), _f64(w)


def _both(A, wf, wc, conj):
    """A w_k (+ conj(A) w_k' where the frequency has a partner)."""
    return A @ wf + (A.conj() @ wc if conj else 0)


def _colloc(case, v, t, W, g=0, keep=None):
    """Y[:, l] = A(s_l) w_l over the kept pairs (all, or the mask's rows), collocation at the centroids."""
    s, _, uniq, part = _s(case, g)
    P, n, area = _panels(v, t)
    c = P.sum(1) / 3.0
    L, wq = _radon7()
    y = torch.einsum("qa,eak->eqk", L, P)                        # quadrature points
    E, dlp = P.shape[0], case["kernel"] == "dlp"
    Y = torch.zeros(E, case["K"], dtype=torch.complex128, device=DEV)
    gx, gw = (_f64(x) for x in np.polynomial.legendre.leggauss(24))
    rows = max(1, 12_000_000 // (7 * E))
    for i0 in range(0, E, rows):
        i = torch.arange(i0, min(E, i0 + rows), device=DEV)
        z = c[i, None, None, :] - y[None]
        r = z.norm(dim=3)
        a = wq * area[None, :, None] / (4 * math.pi * r)
        if dlp:
            a = a * (((c[i, None] - P[None, :, 0]) * n[None]).sum(2)[:, :, None]) / r ** 2
        mask = torch.ones(len(i), E, dtype=torch.bool, device=DEV) if keep is None else keep[i].clone()
        mask[torch.arange(len(i), device=DEV), i] = False
        a = torch.where(mask[:, :, None], a, torch.zeros_like(a))
        for k in uniq:
            x = complex(s[k])
            ph = -x.imag * r
            e = torch.polar(a * torch.exp(-x.real * r), ph)
            A = (e * (1 + x * r) if dlp else e).sum(2)
            Y[i, k] += A @ W[:, k]
            if part[k] != k:
                Y[i, part[k]] += A.conj() @ W[:, part[k]]
    if not dlp:   # self entries: polar coordinates about the centroid, the radial integral in closed form
        for e0 in range(3):
            A_, B_ = P[:, e0] - c, P[:, (e0 + 1) % 3] - c
            u = (B_ - A_) / (B_ - A_).norm(dim=1, keepdim=True)
            t1, t2 = (A_ * u).sum(1), (B_ * u).sum(1)
            d = (A_ - t1[:, None] * u).norm(dim=1)
            p1, p2 = torch.atan2(t1, d), torch.atan2(t2, d)
            rho = d[:, None] / torch.cos(0.5 * (p2 - p1)[:, None] * gx + 0.5 * (p1 + p2)[:, None])
            w = 0.5 * (p2 - p1)[:, None] * gw / (4 * math.pi)
            for k in uniq:
                x = complex(s[k])
                v_ = (w * -torch.expm1(-x * rho) / x).sum(1)
                Y[:, k] += v_ * W[:, k]
                if part[k] != k:
                    Y[:, part[k]] += v_.conj() * W[:, part[k]]
    return Y


def _ss_maps(cas, x, a, b, c):
    """Sauter-Schwab regions: (weight, point of the first panel, of the second)."""
    one = x ** 3 * a ** 2 * b
    if cas == 3:
        h = [((x, x * (1 - a + a * b)), (x * (1 - a * b * c), x * (1 - a))),
             ((x, x * a * (1 - b + b * c)), (x * (1 - a * b), x * a * (1 - b))),
             ((x * (1 - a * b * c), x * a * (1 - b * c)), (x, x * a * (1 - b)))]
        return [(one, p, q) for p, q in h] + [(one, q, p) for p, q in h]
    if cas == 2:
        return [(x ** 3 * a ** 2, (x, x * a * c), (x * (1 - a * b), x * a * (1 - b))),
                (one, (x, x * a), (x * (1 - a * b * c), x * a * b * (1 - c))),
                (one, (x * (1 - a * b), x * a * (1 - b)), (x, x * a * b * c)),
                (one, (x * (1 - a * b * c), x * a * b * (1 - c)), (x, x * a)),
                (one, (x * (1 - a * b * c), x * a * (1 - b * c)), (x, x * a * b))]
    return [(x ** 3 * b, (x, x * a), (x * b, x * b * c)), (x ** 3 * b, (x * b, x * b * c), (x, x * a))]


def _adjacent(t):
    """{1, 2, 3 common vertices: [(first, second, vertex orders of both: the common ones first)]}."""
    at = {}
    for e, tri in enumerate(t.tolist()):
        for p in tri:
            at.setdefault(p, []).append(e)
    out = {1: [], 2: [], 3: []}
    for e, tri in enumerate(t.tolist()):
        for f in sorted({f for p in tri for f in at[p]}):
            o = t[f].tolist()
            sh = [p for p in tri if p in o]
            if len(sh) == 2 and tri.index(sh[1]) - tri.index(sh[0]) == 2:
                sh = sh[::-1]                                    # the edge as it runs in the first panel
            rest = lambda x: [p for p in x if p not in sh]  # noqa: E731
            out[len(sh)].append((e, f, [tri.index(p) for p in sh + rest(tri)], [o.index(p) for p in sh + rest(o)]))
    return out


def _galerkin(case, v, t, W):
    """Y[:, l] = A(s_l) w_l: single layer with constant elements, or the hypersingular operator
    (integrated by parts) with linear ones, on element-local functions (3 per element)."""
    s, _, uniq, part = _s(case)
    P, n, area = _panels(v, t)
    E, hyp = P.shape[0], case["kernel"] == "hyp"
    L, w4 = _conical4()
    w4 = 2.0 * w4 * 0.5
    X = torch.einsum("qa,eak->eqk", L, P)
    Wa = w4[None] * area[:, None]
    T = _f64(t).long()
    nv = v.shape[0]
    Y = torch.zeros(nv if hyp else E, case["K"], dtype=torch.complex128, device=DEV)
    # n x grad of the three barycentric coordinates
    curl = torch.stack([P[:, (b + 2) % 3] - P[:, (b + 1) % 3] for b in range(3)], 1) / (2.0 * area[:, None, None])
    curl = torch.linalg.cross(n[:, None].expand_as(curl), torch.linalg.cross(n[:, None].expand_as(curl), curl))
    adj = _adjacent(t)
    near = torch.zeros(E, E, dtype=torch.bool, device=DEV)
    for k in adj:
        for e, f, _, _ in adj[k]:
            near[e, f] = True

    def add(k, col, vals):
        Y[:, col].index_add_(0, T.reshape(-1), vals.reshape(-1)) if hyp else Y[:, col].add_(vals)

    # regular pairs: a dense product over all points, by rows of elements
    rows = max(1, 3_000_000 // (16 * E))
    Wl = W[T] if hyp else None                                    # [E, 3, K]
    for i0 in range(0, E, rows):
        i = torch.arange(i0, min(E, i0 + rows), device=DEV)
        r = (X[i][:, :, None, None, :] - X[None, None]).norm(dim=4)           # [i, p, E, q]
        a = Wa[i][:, :, None, None] * Wa[None, None] * (~near[i])[:, None, :, None] / (4 * math.pi * r)
        a = torch.where(near[i][:, None, :, None], torch.zeros_like(a), a)
        for k in uniq:
            x = complex(s[k])
            K_ = torch.polar(a * torch.exp(-x.real * r), -x.imag * r)
            for col, M, sx in [(k, K_, x)] + ([(part[k], K_.conj(), x.conjugate())] if part[k] != k else []):
                if not hyp:
                    Y[i, col] += (M.sum(3).sum(1)) @ W[:, col]
                    continue
                wv = Wl[:, :, col]
                M2 = M.reshape(len(i) * 4, E * 4)
                f = torch.einsum("qb,eb->eq", L.to(wv.dtype), wv)             # trial values at the points
                u = torch.einsum("ek,eq->eqk", n.to(wv.dtype), f).reshape(E * 4, 3)
                cu = torch.einsum("ebk,eb->ek", curl.to(wv.dtype), wv)[:, None].expand(E, 4, 3).reshape(E * 4, 3)
                G = (M2 @ torch.cat([u, cu], 1)).reshape(len(i), 4, 6)
                loc = sx * sx * torch.einsum("ik,ipk,pa->ia", n[i].to(wv.dtype), G[:, :, :3], L.to(wv.dtype))
                loc = loc + torch.einsum("iak,ipk->ia", curl[i].to(wv.dtype), G[:, :, 3:])
                Y[:, col].index_add_(0, T[i].reshape(-1), loc.reshape(-1))
    # pairs with a common vertex, edge or panel
    gx, gw = np.polynomial.legendre.leggauss(6)
    g4 = [_f64(z).reshape(-1) for z in np.meshgrid(*[0.5 * (gx + 1)] * 4, indexing="ij")]
    wt = _f64(np.einsum("a,b,c,d->abcd", *[0.5 * gw] * 4)).reshape(-1)
    for cas, pairs in adj.items():
        if not pairs:
            continue
        ei, ej = _f64([p[0] for p in pairs]), _f64([p[1] for p in pairs])
        oi, oj = _f64([p[2] for p in pairs]), _f64([p[3] for p in pairs])
        step = 400
        for q0 in range(0, len(pairs), step):
            i, j, pi, pj = ei[q0:q0 + step], ej[q0:q0 + step], oi[q0:q0 + step], oj[q0:q0 + step]
            A = torch.gather(P[i], 1, pi[:, :, None].expand(-1, -1, 3))
            B = torch.gather(P[j], 1, pj[:, :, None].expand(-1, -1, 3))
            jac = 4.0 * area[i] * area[j] / (4 * math.pi)
            cc = torch.einsum("iak,ibk->iab", torch.gather(curl[i], 1, pi[:, :, None].expand(-1, -1, 3)),
                              torch.gather(curl[j], 1, pj[:, :, None].expand(-1, -1, 3)))
            nn = (n[i] * n[j]).sum(1)
            m = torch.zeros(len(uniq), len(i), 10, dtype=torch.complex128, device=DEV)
            for f, x_, y_ in _ss_maps(cas, *g4):
                bx = torch.stack([1 - x_[0], x_[0] - x_[1], x_[1]], 1)          # barycentric [q, 3]
                by = torch.stack([1 - y_[0], y_[0] - y_[1], y_[1]], 1)
                r = (torch.einsum("qa,iak->iqk", bx, A) - torch.einsum("qa,iak->iqk", by, B)).norm(dim=2)
                h = wt * f * jac[:, None] / r
                phi = torch.cat([torch.ones_like(bx[:, :1]), (bx[:, :, None] * by[:, None]).reshape(-1, 9)], 1)
                if not hyp:
                    phi = phi[:, :1]
                for u, k in enumerate(uniq):
                    x = complex(s[k])
                    m[u, :, :phi.shape[1]] += torch.polar(h * torch.exp(-x.real * r), -x.imag * r) @ phi.to(m.dtype)
            for u, k in enumerate(uniq):
                for col in {int(k), int(part[k])}:
                    sx = complex(s[k]) if col == k else complex(s[k]).conjugate()
                    mm = m[u] if col == k else m[u].conj()
                    if not hyp:
                        Y[:, col].index_add_(0, i, mm[:, 0] * W[j, col])
                        continue
                    blk = cc * mm[:, :1, None] + sx * sx * nn[:, None, None] * mm[:, 1:].reshape(-1, 3, 3)
                    vj = torch.gather(T[j], 1, pj)
                    loc = torch.einsum("iab,ib->ia", blk, W[vj, col])
                    Y[:, col].index_add_(0, torch.gather(T[i], 1, pi).reshape(-1), loc.reshape(-1))
    return Y


#: Evaluations of the kernel above which the 64-bit values would take too long.
MOST = 1.5e10


def exact(case, seed):
    ms, Ws = _inputs(case, seed)
    if case["do"] == "march":
        s, om, _, _ = _s(case)
        x = torch.zeros(Ws[0].shape, dtype=torch.complex128, device=DEV)
        S = _f64(s)[None]
        for n in range(STEPS):
            x = (x + DTS[n] * Ws[0][:, n].to(x.dtype)[:, None]) / (1.0 - DTS[n] * S)
        return {"y": [None] * STEPS, "X": x}
    evals = sum(t.shape[0] ** 2 for _, t in ms) * (16 if case["scheme"] != "colloc7" else 7) * (case["K"] // 2 + 1)
    if evals > MOST:
        return None
    out = []
    for g, ((v, t), W) in enumerate(zip(ms, Ws)):
        W = W.to(torch.complex128)
        keep = None
        if case["do"] == "near":
            perm, blocks = _partition(v, t, case["max_block"])
            keep = np.zeros((t.shape[0],) * 2, dtype=bool)
            for a, b, c, d, far in blocks:
                if not far:
                    keep[np.ix_(perm[a:b], perm[c:d])] = True
            keep = _f64(keep)
        Y = _galerkin(case, v, t, W) if case["scheme"] != "colloc7" else _colloc(case, v, t, W, g, keep)
        y = Y if case["mode"] == "perfreq" else Y.sum(1)
        out.append(y.cpu().numpy() if case["host"] else y)
    return out if case["do"] == "batch" else out[0]
