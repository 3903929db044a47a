"""What the speed of this library is measured on: its public entry points over
the range of maps, batches, footprints and types that programs call them with.

Each case is one call, or one short sequence of calls, of a renderer or a
serving process on a resident map: densities of a batch (`eval`), a frame that
rebuilds an animated map and takes its queries from host memory (`frame`), one
step of a server (`serve`), projected areas (`area`), the cluster hierarchy
(`clusters`) and its cut (`eval` with tau), the GGX fit (`ggx`), and the
per-pixel shading calls (`shade`).

`exact` computes the same results in 64 bits from the definitions: sums over
every triangle in a footprint's window, quadrature of the visible part of each
normal triangle, least squares per node.
"""

import math

import numpy as np
import torch

from paper_2505_08985_gb300 import pndf, synth

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _eval(name, map, n, nq, smin, smax, aspect=1.0, near=0.7, bounds="f16", texels="f32", kernel="gauss", tau=0.0):
    return dict(name=name, kind="eval", map=map, n=n, nq=nq, smin=smin, smax=smax, aspect=aspect, near=near,
                bounds=bounds, texels=texels, kernel=kernel, tau=tau)


def listed():
    return [
        # the smallest everyday call: one tile of a small map, latency and launches
        _eval("bumps256_4k", "bumps", 256, 4096, 4.0, 4.0, near=1.0, bounds="f32"),
        # a 1024^2 image over a scratched map, anisotropic footprints, the plain FP32 path
        _eval("scratch2048_1m", "scratch", 2048, 1 << 20, 1.0, 64.0, aspect=4.0, bounds="f32"),
        # the headline workload: 4M queries on metallic flakes, binary16 bounds
        _eval("flake8192_4m", "flake", 8192, 1 << 22, 1.0, 512.0),
        # few, very large footprints on a 16384^2 binary16 map
        _eval("mixed16384_4k", "mixed", 16384, 4096, 1.0, 1024.0, texels="f16"),
        # a 1024^2 image through the cluster cut (the approximate mode)
        _eval("cut4096_1m", "flake", 4096, 1 << 20, 1.0, 256.0, tau=1e-3),
        # a frame of an animated map: rebuild from device texels, a ragged batch from and to host memory
        dict(name="frame8192_host", kind="frame", map="flake", n=8192, nq=20011, smin=1.0, smax=512.0, bounds="f16",
             texels="f32"),
        # one server step over three maps: ragged camera batches and projected-area requests together
        dict(name="serve_step", kind="serve", b0=1000, b1=9973, b2=37411, b3=65536, areas=16, bounds="f16",
             texels="f32"),
        # diffuse shading under large footprints (the projected area of the mixed map)
        dict(name="area16384_192", kind="area", map="mixed", n=16384, nq=192, smin=1.0, smax=1024.0, texels="f16"),
        # diffuse shading of a tile of a small map
        dict(name="area1024_1k", kind="area", map="scratch", n=1024, nq=1000, smin=1.0, smax=16.0, texels="f32"),
        # building the cluster hierarchy and reading its levels
        dict(name="clusters4096", kind="clusters", map="flake", n=4096, bounds="f16", texels="f32"),
        # fitting the GGX projected area of every mip node
        dict(name="ggx2048", kind="ggx", map="mixed", n=2048, texels="f16"),
        # path-tracer shading: sample a normal and evaluate the shadow-masking per pixel
        dict(name="shade_1m", kind="shade", map="scratch", n=2048, nq=1000003, smin=1.0, smax=64.0, kernel="gauss",
             jac_eps=1e-6, texels="f32"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mean_s2(smin, smax):
    """Mean of sigma^2 for sigma log-uniform in [smin, smax]."""
    return smin * smin if smin == smax else (smax * smax - smin * smin) / (2.0 * math.log(smax / smin))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "eval", "frame", "serve", "area", "area", "clusters", "ggx", "shade"])
    n = int(_log(rng, 64, 8193))
    map = rng.choice(["bumps", "scratch", "flake", "mixed"])
    bounds, texels = rng.choice(["f32", "f16"]), rng.choice(["f32", "f16"])
    smin = 1.0
    smax = _log(rng, 2.0, max(4.0, n / 16.0))
    if kind == "eval":
        nq = min(int(_log(rng, 1, 1 << 22)), int(8e9 / _mean_s2(smin, smax)))
        what = rng.choice(["gauss", "gauss", "gauss", "disk", "box", "clamp", "cut"])
        c = _eval("", map, n, max(1, nq), smin, smax, aspect=rng.uniform(1.0, 4.0), near=rng.uniform(0.5, 1.0),
                  bounds=bounds, texels=texels, kernel="gauss" if what == "cut" else what,
                  tau=_log(rng, 1e-4, 1e-1) if what == "cut" else 0.0)
        del c["name"]
        return c
    if kind == "frame":
        nq = min(int(_log(rng, 1, 1 << 17)), int(1e9 / _mean_s2(smin, smax)))
        return dict(kind=kind, map=map, n=n, nq=max(1, nq), smin=smin, smax=smax, bounds=bounds, texels=texels)
    if kind == "serve":
        return dict(kind=kind, b0=int(_log(rng, 1, 1e5)), b1=int(_log(rng, 1, 1e5)), b2=int(_log(rng, 1, 1e5)),
                    b3=int(_log(rng, 1, 1e5)), areas=rng.randrange(0, 33), bounds=bounds, texels=texels)
    if kind == "area":
        nq = min(int(_log(rng, 1, 1 << 14)), int(2e7 / _mean_s2(smin, smax)))
        return dict(kind=kind, map=map, n=n, nq=max(1, nq), smin=smin, smax=smax, texels=texels)
    if kind == "clusters":
        return dict(kind=kind, map=map, n=min(n, 4096), bounds=bounds, texels=texels)
    if kind == "ggx":
        return dict(kind=kind, map=map, n=min(n, 2048), texels=texels)
    return dict(kind=kind, map=map, n=min(n, 2048), nq=int(_log(rng, 1, 1 << 20)), smin=smin, smax=smax,
                kernel=rng.choice(["gauss", "disk", "box"]), jac_eps=rng.choice([0.0, 1e-6]), texels=texels)


# ---------------------------------------------------------------------------
# inputs and state
# ---------------------------------------------------------------------------

def _map(kind, n, texels, seed):
    """The normal maps of the library's workloads: feature counts per area as in the full-size ones."""
    area = n * n
    if kind == "bumps":
        st = synth.bumps_map(n=n, n_bumps=max(1, area // 1024), seed=seed, device=DEV) if n <= 1024 else \
            synth.normals_from_height(synth.value_noise(n, seed, DEV, base_period=32, amplitude=4.0))
    elif kind == "scratch":
        st = synth.scratch_map(n=n, n_grooves=min(2000, max(1, area // 2097)), seed=seed, device=DEV)
    elif kind == "flake":
        st = synth.flake_map(n=n, n_cells=max(4, area // 336), seed=seed, device=DEV)
    else:
        st = synth.mixed_map(n=n, n_cells=max(4, area // 336), n_grooves=min(2000, max(1, area // 33554)), seed=seed,
                             device=DEV)
    return st.half() if texels == "f16" else st


def _queries(st, case, seed):
    mix = synth.QueryMix(sigma=(case["smin"], case["smax"]), aspect=(1.0, case.get("aspect", 1.0)),
                         frac_near=case.get("near", 0.7))
    return synth.make_queries(st, case["nq"], mix, seed)


SERVE_MAPS = (("bumps", 1024), ("scratch", 2048), ("flake", 4096))


def _inputs(case, seed):
    """Everything the case reads, made from the seed alone."""
    kind = case["kind"]
    if kind == "serve":
        sts = [_map(m, n, case["texels"], 10 * seed + k) for k, (m, n) in enumerate(SERVE_MAPS)]
        on = [(k + seed) % 3 for k in range(4)]
        qs = [synth.camera_queries(SERVE_MAPS[on[k]][1], case["b%d" % k], 10 * seed + k, device=DEV) for k in range(4)]
        aq = synth.make_queries(sts[1], max(1, case["areas"]), synth.QueryMix(sigma=(1.0, 32.0)), seed)
        w = synth.hemisphere_dirs(max(1, case["areas"]), seed, DEV)
        return dict(sts=sts, on=on, qs=qs, aq=aq, w=w)
    st = _map(case["map"], case["n"], case["texels"], seed)
    out = dict(st=st)
    if "nq" in case:
        out["q"] = _queries(st, case, seed)
    if kind == "area":
        out["w"] = synth.hemisphere_dirs(case["nq"], seed, DEV)
    if kind == "shade":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        out["u"] = torch.rand(case["nq"], 2, generator=g, device=DEV)
        out["wi"] = synth.hemisphere_dirs(case["nq"], seed + 1, DEV, min_z=0.05)
        out["wo"] = synth.hemisphere_dirs(case["nq"], seed + 2, DEV, min_z=0.05)
    return out


BOUNDS = {"f32": pndf.PNDF_BOUNDS_F32, "f16": pndf.PNDF_BOUNDS_F16_OUTWARD}
KERNELS = {"gauss": pndf.PNDF_KERNEL_GAUSS, "disk": pndf.PNDF_KERNEL_DISK, "box": pndf.PNDF_KERNEL_BOX,
           "clamp": pndf.PNDF_KERNEL_GAUSS}


def prepare(case, seed):
    """The resident map(s) and the batch in the caller's hands; nothing is evaluated here."""
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    bounds = BOUNDS[case.get("bounds", "f16")]
    if kind == "serve":
        s["hs"] = [pndf.pndf_build_hierarchy(st, bounds_fmt=bounds) for st in s.pop("sts")]
        s["srv"] = pndf.pndf_server_create(s["hs"], max_segments=16, max_area_requests=64)
        s["D"] = [torch.empty(q.shape[0], device=DEV) for q in s["qs"]]
        s["P"] = torch.empty(s["aq"].shape[0], device=DEV)
        return s
    h = pndf.pndf_build_hierarchy(s["st"], bounds_fmt=bounds, clusters=kind == "clusters" or case.get("tau", 0.0) > 0)
    s["h"] = h
    if kind == "eval":
        s["out"] = torch.empty(case["nq"], device=DEV)
    if kind == "frame":
        s["q"] = s["q"].cpu().pin_memory()
        s["out"] = torch.empty(case["nq"], pin_memory=True)
    if kind == "shade":
        s["g"] = pndf.pndf_ggx_create(h)
    if kind not in ("frame", "clusters"):
        del s["st"]
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "eval":
        if case["kernel"] == "gauss" and case["tau"] == 0.0:
            return pndf.pndf_eval_batch(s["h"], s["q"], out=s["out"])
        return pndf.pndf_eval_batch_ex(s["h"], s["q"], out=s["out"], kernel=KERNELS[case["kernel"]], tau=case["tau"],
                                       jac_eps=1e-6 if case["kernel"] == "clamp" else 0.0)
    if kind == "frame":
        pndf.pndf_update_hierarchy(s["h"], s["st"])
        return pndf.pndf_eval_batch_host(s["h"], s["q"], s["out"])
    if kind == "serve":
        segs = [(s["on"][k], q, None, s["D"][k], None, 0, q.shape[0]) for k, q in enumerate(s["qs"])]
        if case["areas"]:
            segs.append((1, s["aq"], None, s["P"], None, 0, case["areas"], pndf.PNDF_SEGMENT_PROJECTED_AREA, s["w"]))
        pndf.pndf_server_step(s["srv"], segs)
        return s["D"] + ([s["P"]] if case["areas"] else [])
    if kind == "area":
        return pndf.pndf_diffuse_projected_area(s["h"], s["q"], s["w"])
    if kind == "clusters":
        pndf.pndf_update_hierarchy(s["h"], s["st"])
        return [pndf.pndf_cluster_level(s["h"], level) for level in range(2, pndf.top_level(case["n"]) + 1)]
    if kind == "ggx":
        g = pndf.pndf_ggx_create(s["h"])
        return [pndf.pndf_ggx_level(g, level) for level in range(2, pndf.top_level(case["n"]) + 1)]
    m, tri, flags = pndf.pndf_sample_normals(s["h"], s["q"], s["u"], kernel=KERNELS[case["kernel"]],
                                             jac_eps=case["jac_eps"])
    return m, tri, flags, pndf.pndf_shadow_masking(s["g"], s["q"], s["wi"], s["wo"])


def work(case):
    """Inputs read once (texels, queries, directions), results written once;
    operations: the triangles that have to be integrated, the least squares."""
    kind = case["kind"]
    if kind == "serve":
        nq = sum(case["b%d" % k] for k in range(4))
        tex = sum(n * n for _, n in SERVE_MAPS) * (4 if case["texels"] == "f16" else 8)
        return dict(bytes=float(min(tex, 8 * 1000.0 * nq) + 36 * nq + 48 * case["areas"]),
                    flops=60.0 * 2 * 16 * math.pi * _mean_s2(1.0, 32.0) * case["areas"])
    n2 = float(case["n"]) ** 2
    tb = 4 if case["texels"] == "f16" else 8
    nq = case.get("nq", 0)
    quads = 16 * math.pi * _mean_s2(case["smin"], case["smax"]) * nq if nq else 0.0  # in the footprints
    levels = n2 / 16 * 4 / 3
    if kind == "eval":  # a density reads at most the texels its footprints cover
        return dict(bytes=min(n2, quads) * tb + 36.0 * nq, flops=50.0 * nq)
    if kind == "frame":
        return dict(bytes=n2 * tb + 36.0 * nq, flops=50.0 * nq)
    if kind == "area":
        return dict(bytes=min(n2, quads) * tb + 48.0 * nq, flops=60.0 * 2 * min(quads, n2 * nq))
    if kind == "clusters":
        return dict(bytes=n2 * tb + levels * 36, flops=2000.0 * levels)
    if kind == "ggx":
        return dict(bytes=n2 * tb + levels * 12, flops=2 * n2 * (60 + 16 * 4) + levels * 96)
    return dict(bytes=min(n2, 4.0 * nq) * tb + nq * (32 + 8 + 24 + 16 + 4.0), flops=200.0 * nq)


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

CHUNK = 1 << 23  # quads of footprint windows in hand at once


def _windows(q, n, r):
    """Quad windows [i0, i1] x [j0, j1] of the footprints' half-widths r = (rx, ry)."""
    x, y = q[:, 0].to(F64), q[:, 1].to(F64)
    lo = torch.stack((x - r[0], y - r[1]), 1).floor() - 1
    hi = torch.stack((x + r[0], y + r[1]), 1).ceil() + 1
    lo, hi = lo.clamp(0, n - 1).long(), hi.clamp(-1, n - 2).long()
    return lo, (hi - lo + 1).clamp(min=0)


def _window_chunks(q, n, r):
    """Chunks (query index, i, j) covering every quad of every window once."""
    lo, size = _windows(q, n, r)
    total = (size[:, 0] * size[:, 1]).cpu().numpy()
    order = np.argsort(total, kind="stable")
    k = 0
    while k < len(order):
        if total[order[k]] == 0:
            k += 1
            continue
        if total[order[k]] >= CHUNK:  # one large window, by rows
            t = int(order[k])
            (i0, j0), (w, hgt) = lo[t].tolist(), size[t].tolist()
            rows = max(1, CHUNK // w)
            for r0 in range(0, hgt, rows):
                jj = torch.arange(j0 + r0, j0 + min(hgt, r0 + rows), device=DEV)
                ii = torch.arange(i0, i0 + w, device=DEV)
                j, i = torch.meshgrid(jj, ii, indexing="ij")
                yield torch.full((i.numel(),), t, device=DEV), i.reshape(-1), j.reshape(-1)
            k += 1
            continue
        # many small windows: as many as fit
        e = min(len(order), k + max(1, int(CHUNK // total[order[k]])))
        while int(total[order[k:e]].sum()) > CHUNK:
            e = k + max(1, (e - k) // 2)
        t = torch.from_numpy(order[k:e]).to(DEV)
        cnt = torch.from_numpy(total[order[k:e]]).to(DEV)
        qi = torch.repeat_interleave(t, cnt)
        at = torch.arange(qi.numel(), device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
        w = size[qi, 0]
        yield qi, lo[qi, 0] + at % w, lo[qi, 1] + at // w
        k = e


def _texel(st, i, j):
    return st[j, i].to(F64)


def _cross(a, b):
    return a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]


def _exact_pndf(st, q, kernel):
    """Eq. 5 by exhaustion over the windows; kernel 'clamp' is Eq. 6 with eps 1e-6."""
    st = st.float()
    n = st.shape[0]
    q64 = q.to(F64)
    sxx, sxy, syy = q64[:, 2], q64[:, 3], q64[:, 4]
    det = sxx * syy - sxy * sxy
    reach = 4.0 if kernel in ("gauss", "clamp") else 1.5
    l21, l22 = sxy / sxx.sqrt(), (syy - sxy * sxy / sxx).clamp(min=0).sqrt()
    ry = reach * ((l21.abs() + l22) if kernel == "box" else syy.sqrt())
    norm = 1.0 / ({"gauss": 2 * math.pi, "clamp": 2 * math.pi, "disk": 2.25 * math.pi, "box": 9.0}[kernel] * det.sqrt())
    rho = math.sqrt(2e-6 / math.sqrt(3.0)) / math.sqrt(3.0) if kernel == "clamp" else 0.0
    corners = torch.stack((st[:-1, :-1], st[:-1, 1:], st[1:, :-1], st[1:, 1:]))
    box = torch.cat((corners.amin(0), -corners.amax(0)), 2).reshape(-1, 4) - 2 * rho
    del corners
    m = torch.cat((q[:, 5:7], -q[:, 5:7]), 1).float()
    D = torch.zeros(q.shape[0], dtype=F64, device=DEV)
    for qi, i, j in _window_chunks(q, n, (reach * sxx.sqrt(), ry)):
        near = (box[j * (n - 1) + i] <= m[qi]).all(1).nonzero()[:, 0]
        qi, i, j = qi[near], i[near], j[near]
        for tri in (0, 1):
            a = _texel(st, i + tri, j + tri)
            b = _texel(st, i + 1 - tri, j + tri)
            c = _texel(st, i + tri, j + 1 - tri)
            p = q64[qi, 5:7]
            cr = _cross(b - a, c - a)
            if rho:
                small = cr.abs() < float(np.float32(1e-6))
                g = (a + b + c) / 3.0
                h = 0.5 * math.sqrt(3.0) * rho
                a = torch.where(small[:, None], g + torch.tensor([0.0, rho], dtype=F64, device=DEV), a)
                b = torch.where(small[:, None], g + torch.tensor([-h, -0.5 * rho], dtype=F64, device=DEV), b)
                c = torch.where(small[:, None], g + torch.tensor([h, -0.5 * rho], dtype=F64, device=DEV), c)
                cr = _cross(b - a, c - a)
            s = torch.sign(cr)
            e0, e1, e2 = _cross(c - b, p - b) * s, _cross(a - c, p - c) * s, _cross(b - a, p - a) * s
            hit = ((s != 0) & (e0 >= 0) & (e1 >= 0) & (e2 >= 0)).nonzero()[:, 0]
            t, acr = qi[hit], cr[hit].abs()
            way = 1 - 2 * tri
            dx = (i[hit] + tri).to(F64) - q64[t, 0] + way * e1[hit] / acr
            dy = (j[hit] + tri).to(F64) - q64[t, 1] + way * e2[hit] / acr
            qq = (syy[t] * dx * dx - 2 * sxy[t] * dx * dy + sxx[t] * dy * dy) / det[t]
            if kernel in ("gauss", "clamp"):
                w = torch.where(qq <= 16.0, torch.exp(-0.5 * qq), 0.0)
            elif kernel == "disk":
                w = (qq <= 2.25).to(F64)
            else:
                v1 = dx * dx / sxx[t]
                w = ((v1 <= 2.25) & (qq - v1 <= 2.25)).to(F64)
            D.index_add_(0, t, norm[t] * w / acr)
    return D


def _gauss(k):
    x, w = np.polynomial.legendre.leggauss(k)
    return torch.tensor(0.5 * (x + 1), dtype=F64, device=DEV), torch.tensor(0.5 * w, dtype=F64, device=DEV)


def _g(w, x, y):
    """max(w . m~, 0) / m~_z at m = (x, y)."""
    z = (1.0 - x * x - y * y).clamp(min=1e-300).sqrt()
    return (w[2] + (w[0] * x + w[1] * y) / z).clamp(min=0.0)


def _duffy(a, b, c, w, k):
    """Half the mean of g over triangles where it is smooth, k x k Gauss points."""
    t, wt = _gauss(k)
    out = torch.zeros(a.shape[0], dtype=F64, device=DEV)
    for u, wu in zip(t.tolist(), wt.tolist()):
        p, d = a + u * (b - a), u * (c - b)
        for v, wv in zip(t.tolist(), wt.tolist()):
            out += (wu * wv * u) * _g(w, p[:, 0] + v * d[:, 0], p[:, 1] + v * d[:, 1])
    return out


def _clip(P, D):
    """Visible interval of the segments P + t D in the frame where the visible
    normals are X >= 0 or X^2 + Y^2 <= 1 (a convex set there); empty: t1 < t0."""
    Q = P + D
    vp = (P[0] >= 0) | (P[0] ** 2 + P[1] ** 2 <= 1)
    vq = (Q[0] >= 0) | (Q[0] ** 2 + Q[1] ** 2 <= 1)
    dd = (D[0] ** 2 + D[1] ** 2).clamp(min=1e-300)
    along, across = P[0] * D[0] + P[1] * D[1], P[0] * D[1] - P[1] * D[0]
    h2 = dd - across * across
    half = h2.clamp(min=0).sqrt()
    tn, tf = (-along - half) / dd, (-along + half) / dd
    zero, one = torch.zeros_like(tn), torch.ones_like(tn)
    inside = (h2 > 0) & (tn >= 0) & (tf <= 1)
    t0 = torch.where(vp, zero, torch.where(vq, tn.clamp(0, 1), torch.where(inside, tn, one)))
    t1 = torch.where(vq, one, torch.where(vp, tf.clamp(0, 1), torch.where(inside, tf, zero)))
    return t0, t1


def _partial(a, b, c, w):
    """Half the mean of g over triangles that are visible in part: lines
    parallel to b - c swept from a, each line clipped exactly, the sweep cut
    where a line's ends cross the visibility boundary or touch it."""
    wr = (w[0] ** 2 + w[1] ** 2).sqrt().clamp(min=1e-300)
    cs, sn = w[0] / wr, w[1] / wr

    def frame(m):
        return torch.stack(((cs * m[:, 0] + sn * m[:, 1]) / w[2], cs * m[:, 1] - sn * m[:, 0]))

    A, B, C = frame(a), frame(b), frame(c)
    E = C - B
    cuts = []
    for D in (B - A, C - A):
        dd = (D[0] ** 2 + D[1] ** 2).clamp(min=1e-300)
        along, across = A[0] * D[0] + A[1] * D[1], A[0] * D[1] - A[1] * D[0]
        half = (dd - across * across).clamp(min=0).sqrt()
        cuts += [(-along - half) / dd, (-along + half) / dd]
    k0, k1 = A[0] * E[1] - A[1] * E[0], (B - A)[0] * E[1] - (B - A)[1] * E[0]
    len_e = (E[0] ** 2 + E[1] ** 2).sqrt()
    k1 = torch.where(k1.abs() < 1e-300, torch.full_like(k1, 1e-300), k1)
    cuts += [(len_e - k0) / k1, (-len_e - k0) / k1]
    zero = torch.zeros_like(len_e)
    cuts = torch.stack([zero, zero + 1] + [t.nan_to_num(0.0).clamp(0, 1) for t in cuts]).sort(0).values
    t, wt = _gauss(12)
    v, wv = _gauss(8)
    out = torch.zeros_like(zero)
    for piece in range(7):
        live = (cuts[piece + 1] > cuts[piece]).nonzero()[:, 0]
        if live.numel() == 0:
            continue
        lo, ln = cuts[piece][live], (cuts[piece + 1] - cuts[piece])[live]
        al, bl, cl, wl = a[live], b[live], c[live], w[:, live]
        Al, Bl, El = A[:, live], B[:, live], E[:, live]
        acc = torch.zeros_like(lo)
        for s, ws in zip(t.tolist(), wt.tolist()):
            tau = lo + ln * (s * s * (3 - 2 * s))
            t0, t1 = _clip(Al + tau * (Bl - Al), tau * El)
            seg = (t1 - t0).clamp(min=0)
            px, py = al[:, 0] + tau * (bl - al)[:, 0], al[:, 1] + tau * (bl - al)[:, 1]
            ex, ey = tau * (cl - bl)[:, 0], tau * (cl - bl)[:, 1]
            inner = torch.zeros_like(lo)
            for u, wu in zip(v.tolist(), wv.tolist()):
                x = t0 + u * seg
                inner += wu * _g(wl, px + x * ex, py + x * ey)
            acc += (ws * 6 * s * (1 - s)) * tau * seg * inner
        out[live] += ln * acc
    return out


def _visible(a, b, c, w):
    """Half the mean of g over each triangle (uv area 1/2); w: (3, count) unit directions."""
    out = torch.zeros(a.shape[0], dtype=F64, device=DEV)

    def v(p):
        return w[0] * p[:, 0] + w[1] * p[:, 1] + w[2] * (1 - (p * p).sum(1)).clamp(min=0).sqrt()

    va, vb, vc = v(a), v(b), v(c)
    full = (va >= 0) & (vb >= 0) & (vc >= 0)
    spread = torch.maximum(((b - a) ** 2).sum(1), torch.maximum(((c - a) ** 2).sum(1), ((c - b) ** 2).sum(1)))
    for lo, hi, k in ((-1.0, 1e-3, 3), (1e-3, 4e-2, 5), (4e-2, 9.0, 9)):
        at = (full & (spread > lo) & (spread <= hi)).nonzero()[:, 0]
        if at.numel():
            out[at] = _duffy(a[at], b[at], c[at], w[:, at], k)
    # concavity: z lies within spread / (6 z^3) of its linear interpolant
    zmin = (1 - torch.maximum((a * a).sum(1), torch.maximum((b * b).sum(1), (c * c).sum(1)))).clamp(min=1e-3).sqrt()
    some = torch.maximum(va, torch.maximum(vb, vc)) + w[2] * spread / (6 * zmin ** 3) >= 0
    at = (~full & some).nonzero()[:, 0]
    if at.numel():
        out[at] = _partial(a[at], b[at], c[at], w[:, at])
    return out


def _exact_area(st, q, w):
    st = st.float()
    n = st.shape[0]
    q64 = q.to(F64)
    sxx, sxy, syy = q64[:, 2], q64[:, 3], q64[:, 4]
    det = sxx * syy - sxy * sxy
    norm = 1.0 / (2 * math.pi * det.sqrt())
    w64 = w.to(F64)
    w64 = w64 / w64.norm(dim=1, keepdim=True)
    P = torch.zeros(q.shape[0], dtype=F64, device=DEV)
    for qi, i, j in _window_chunks(q, n, (4 * sxx.sqrt(), 4 * syy.sqrt())):
        for tri in (0, 1):
            f = (1 + tri) / 3.0
            dx, dy = i.to(F64) + f - q64[qi, 0], j.to(F64) + f - q64[qi, 1]
            qq = (syy[qi] * dx * dx - 2 * sxy[qi] * dx * dy + sxx[qi] * dy * dy) / det[qi]
            at = (qq <= 16.0).nonzero()[:, 0]
            t, ia, ja = qi[at], i[at], j[at]
            val = _visible(_texel(st, ia + tri, ja + tri), _texel(st, ia + 1 - tri, ja + tri),
                           _texel(st, ia + tri, ja + 1 - tri), w64[t].T.contiguous())
            P.index_add_(0, t, norm[t] * torch.exp(-0.5 * qq[at]) * val)
    return P


def _height(n):
    L = 2
    while (1 << L) < n - 1:
        L += 1
    return L


def _nan_outside(v, n, level):
    """(NaN, 0, 0) in the nodes of `level` with a quad outside the map; v: (S, S, 3) indexed [J, I]."""
    inside = (n - 1) >> level
    none = torch.tensor([float("nan"), 0.0, 0.0], dtype=F64, device=DEV)
    v[inside:] = none
    v[:, inside:] = none
    return v


def _exact_ggx(st):
    """Omega per node and level: least squares over 16 directions at w_z = 0.3."""
    st = st.float()
    n = st.shape[0]
    L = _height(n)
    wz = float(np.float32(0.3))
    r = math.sqrt(1 - wz * wz)
    dirs = np.array([[r * math.cos(2 * math.pi * k / 16), r * math.sin(2 * math.pi * k / 16), wz] for k in range(16)])
    dirs = dirs.astype(np.float32).astype(np.float64)
    # per-quad projected area at each direction, padded to the pyramid's side
    S = 1 << (L - 2)
    leaf = torch.zeros(S, S, 16, dtype=F64, device=DEV)
    jj, ii = torch.meshgrid(torch.arange(n - 1, device=DEV), torch.arange(n - 1, device=DEV), indexing="ij")
    ii, jj = ii.reshape(-1), jj.reshape(-1)
    for k in range(16):
        w = torch.tensor(dirs[k], dtype=F64, device=DEV)
        w = w / w.norm()
        for p in range(0, ii.numel(), CHUNK):
            i, j = ii[p:p + CHUNK], jj[p:p + CHUNK]
            wk = w[:, None].expand(3, i.numel()).contiguous()
            for tri in (0, 1):
                v = _visible(_texel(st, i + tri, j + tri), _texel(st, i + 1 - tri, j + tri),
                             _texel(st, i + tri, j + 1 - tri), wk)
                leaf.view(-1).index_add_(0, ((j >> 2) * S + (i >> 2)) * 16 + k, v / 16.0)
    rows = torch.tensor(np.stack((dirs[:, 0] ** 2, 2 * dirs[:, 0] * dirs[:, 1], dirs[:, 1] ** 2), 1), dtype=F64,
                        device=DEV)
    fit = torch.linalg.pinv(rows)
    out = []
    for level in range(2, L + 1):
        a = (2 * leaf - wz) ** 2 - wz * wz
        out.append(_nan_outside(a @ fit.T, n, level))
        leaf = 0.25 * (leaf[0::2, 0::2] + leaf[1::2, 0::2] + leaf[0::2, 1::2] + leaf[1::2, 1::2]) if level < L else leaf
    return out


def _exact_clusters(st):
    """Eq. 7-8 per node, directly from its fine triangles at every level."""
    st = st.float()
    n = st.shape[0]
    L = _height(n)
    side = 1 << L
    pad = torch.zeros(side + 1, side + 1, 2, dtype=F64, device=DEV)
    pad[:n, :n] = st.to(F64)
    inside = torch.zeros(side, side, dtype=F64, device=DEV)
    inside[:n - 1, :n - 1] = 1.0
    off = (((0, 0), (1, 0), (0, 1)), ((1, 1), (0, 1), (1, 0)))  # vertex offsets (x, y)
    wt = []
    for tri in (0, 1):
        a, b, c = (pad[dy:dy + side, dx:dx + side] for dx, dy in off[tri])
        cr = (b[..., 0] - a[..., 0]) * (c[..., 1] - a[..., 1]) - (b[..., 1] - a[..., 1]) * (c[..., 0] - a[..., 0])
        wt.append(inside / cr.abs().clamp(min=1e-6) / 24.0)
    out = []
    for level in range(2, L + 1):
        m = 1 << level
        S = side // m
        y, x = torch.meshgrid(torch.arange(m, device=DEV, dtype=F64), torch.arange(m, device=DEV, dtype=F64),
                              indexing="ij")

        def hats(tri):
            """(3 vertices, 4 hats, m, m): the node's hats at the triangle's vertices."""
            low = (x + y <= m - 1 - tri)[None]
            res = []
            for dx, dy in off[tri]:
                s, t = (x + dx) / m, (y + dy) / m
                lo = torch.stack((1 - s - t, s, t, torch.zeros_like(s)))
                up = torch.stack((torch.zeros_like(s), 1 - t, 1 - s, s + t - 1))
                res.append(torch.where(low, lo, up))
            return torch.stack(res)

        def blocks(v):
            return v.reshape(S, m, S, m).sum((1, 3)).reshape(-1)

        def tile(cst):
            return cst.repeat(S, S)

        G = torch.zeros(S * S, 4, 4, dtype=F64, device=DEV)
        R = torch.zeros(S * S, 4, 2, dtype=F64, device=DEV)
        for tri in (0, 1):
            h = hats(tri)
            hs = h.sum(0)
            nv = [pad[dy:dy + side, dx:dx + side] for dx, dy in off[tri]]
            ns = nv[0] + nv[1] + nv[2]
            for p in range(4):
                for r in range(p, 4):
                    cst = h[0, p] * h[0, r] + h[1, p] * h[1, r] + h[2, p] * h[2, r] + hs[p] * hs[r]
                    if bool((cst != 0).any()):
                        G[:, p, r] += blocks(wt[tri] * tile(cst))
                for ch in (0, 1):
                    v = tile(hs[p]) * ns[..., ch]
                    for k in range(3):
                        v += tile(h[k, p]) * nv[k][..., ch]
                    R[:, p, ch] += blocks(wt[tri] * v)
        # symmetric elimination, unrolled over the 4 x 4 system
        for p in range(4):
            for r in range(p):
                G[:, p, r] = G[:, r, p]
        ok = (torch.arange(S, device=DEV) < ((n - 1) >> level)).to(F64)
        ok = (ok[:, None] * ok[None, :]).reshape(-1) > 0
        G[~ok] = torch.eye(4, dtype=F64, device=DEV)
        M = torch.cat((G, R), 2)
        for p in range(4):
            M[:, p] = M[:, p] / M[:, p, p:p + 1]
            for r in range(4):
                if r != p:
                    M[:, r] = M[:, r] - M[:, r, p:p + 1] * M[:, p]
        cor = M[:, :, 4:]
        F = torch.zeros(S * S, dtype=F64, device=DEV)
        for tri in (0, 1):
            h = hats(tri)
            nv = [pad[dy:dy + side, dx:dx + side] for dx, dy in off[tri]]
            for ch in (0, 1):
                field = cor[:, :, ch].reshape(S, S, 4)
                tot, sq = 0.0, 0.0
                for k in range(3):
                    fit = torch.einsum("jia,ayx->jyix", field, h[k]).reshape(side, side)
                    dlt = fit - nv[k][..., ch]
                    tot, sq = tot + dlt, sq + dlt * dlt
                F += blocks(wt[tri] * (sq + tot * tot))
        rec = torch.cat((cor[:, 0], cor[:, 1] - cor[:, 0], cor[:, 2] - cor[:, 0], cor[:, 3] - cor[:, 0]), 1)
        rec[~ok] = 0.0
        e = F.clamp(min=0).sqrt()
        e[~ok] = float("inf")
        out.append((rec.reshape(S, S, 8), e.reshape(S, S)))
    return out


def _exact_samples(st, q, u, kernel, eps):
    st = st.float()
    n = st.shape[0]
    q64, u64 = q.to(F64), u.to(F64)
    if kernel == "box":
        v = 1.5 * (2 * u64 - 1)
    else:
        rad = 1.5 * u64[:, 0].sqrt() if kernel == "disk" else \
            (-2.0 * torch.log(1.0 - u64[:, 0] * (1.0 - math.exp(-8.0)))).sqrt()
        ang = 2 * math.pi * u64[:, 1]
        v = torch.stack((rad * ang.cos(), rad * ang.sin()), 1)
    l11 = q64[:, 2].sqrt()
    l21 = q64[:, 3] / l11
    l22 = (q64[:, 4] - l21 * l21).sqrt()
    px, py = q64[:, 0] + l11 * v[:, 0], q64[:, 1] + l21 * v[:, 0] + l22 * v[:, 1]
    i, j = px.floor(), py.floor()
    ok = (i >= 0) & (j >= 0) & (i <= n - 2) & (j <= n - 2)
    fu, fv = px - i, py - j
    i, j = torch.where(ok, i, 0.0).long(), torch.where(ok, j, 0.0).long()
    tri = (fu + fv >= 1.0).long()
    a, b, c = _texel(st, i + tri, j + tri), _texel(st, i + 1 - tri, j + tri), _texel(st, i + tri, j + 1 - tri)
    up = tri > 0
    l0 = torch.where(up, fu + fv - 1, 1 - fu - fv)
    lb, lc = torch.where(up, 1 - fu, fu), torch.where(up, 1 - fv, fv)
    if eps > 0:
        eps = float(np.float32(eps))
        small = (_cross(b - a, c - a).abs() < eps)[:, None]
        rho = math.sqrt(2 * eps / math.sqrt(3.0)) / math.sqrt(3.0)
        h = 0.5 * math.sqrt(3.0) * rho
        g = (a + b + c) / 3.0
        a = torch.where(small, g + torch.tensor([0.0, rho], dtype=F64, device=DEV), a)
        b = torch.where(small, g + torch.tensor([-h, -0.5 * rho], dtype=F64, device=DEV), b)
        c = torch.where(small, g + torch.tensor([h, -0.5 * rho], dtype=F64, device=DEV), c)
    return torch.where(ok[:, None], l0[:, None] * a + lb[:, None] * b + lc[:, None] * c, 0.0)


def _exact_masking(st, q, wi, wo):
    """The height-correlated G of Sec. 4.3 from the nodes' Omega, two mip levels bilinear."""
    n = st.shape[0]
    L = _height(n)
    omega = _exact_ggx(st)
    q64, wi, wo = q.to(F64), wi.to(F64), wo.to(F64)
    lam = torch.log2(math.sqrt(12.0) * torch.maximum(q64[:, 2], q64[:, 4]).sqrt()).clamp(2.0, float(L))
    l0 = lam.floor().long()
    O = torch.zeros(q.shape[0], 3, dtype=F64, device=DEV)
    wsum = torch.zeros(q.shape[0], dtype=F64, device=DEV)
    for side in (0, 1):
        for level in range(2, L + 1):
            at = ((l0 if side == 0 else (l0 + 1).clamp(max=L)) == level).nonzero()[:, 0]
            if at.numel() == 0:
                continue
            wl = lam[at] - l0[at].to(F64)
            wl = wl if side else 1 - wl
            S = omega[level - 2].shape[0]
            f = q64[at, :2] / float(1 << level) - 0.5
            fl = f.floor()
            part = torch.zeros(at.numel(), 3, dtype=F64, device=DEV)
            pw = torch.zeros(at.numel(), dtype=F64, device=DEV)
            for dj in (0, 1):
                for di in (0, 1):
                    I = (fl[:, 0] + di).clamp(0, S - 1).long()
                    J = (fl[:, 1] + dj).clamp(0, S - 1).long()
                    o = omega[level - 2][J, I]
                    t = f - fl
                    w = (t[:, 0] if di else 1 - t[:, 0]) * (t[:, 1] if dj else 1 - t[:, 1])
                    w = torch.where(o[:, 0].isfinite(), w, 0.0)
                    part += w[:, None] * o.nan_to_num(0.0)
                    pw += w
            use = torch.where(pw > 0, wl, 0.0)
            O[at] += (use / pw.clamp(min=1e-300))[:, None] * part
            wsum[at] += use
    good = wsum > 0
    O = O / wsum.clamp(min=1e-300)[:, None]

    def lam_of(w):
        qf = O[:, 0] * w[:, 0] ** 2 + 2 * O[:, 1] * w[:, 0] * w[:, 1] + O[:, 2] * w[:, 1] ** 2
        return 0.5 * (w[:, 2] + (w[:, 2] ** 2 + qf).clamp(min=0).sqrt()) / w[:, 2] - 1

    m = q64[:, 5:7]
    mz = (1 - (m * m).sum(1)).clamp(min=0).sqrt()
    ci = (m * wi[:, :2]).sum(1) + mz * wi[:, 2]
    co = (m * wo[:, :2]).sum(1) + mz * wo[:, 2]
    G = torch.where((ci > 0) & (co > 0), 1.0 / (1.0 + lam_of(wi) + lam_of(wo)), 0.0)
    return torch.where(good, G, float("nan"))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("eval", "frame"):
        # the cut's result is defined by rounded records; the largest batches take minutes
        if case.get("tau", 0.0) > 0 or 64.0 * _mean_s2(case["smin"], case["smax"]) * case["nq"] > 4e10:
            return None
        s = _inputs(case, seed)
        return _exact_pndf(s["st"], s["q"], case.get("kernel", "gauss"))
    if kind == "area":
        s = _inputs(case, seed)
        return _exact_area(s["st"], s["q"], s["w"])
    if kind == "serve":
        s = _inputs(case, seed)
        out = [_exact_pndf(s["sts"][s["on"][k]], q, "gauss") for k, q in enumerate(s["qs"])]
        return out + ([_exact_area(s["sts"][1], s["aq"][:case["areas"]], s["w"])] if case["areas"] else [])
    s = _inputs(case, seed)
    if kind == "clusters":
        return _exact_clusters(s["st"])
    if kind == "ggx":
        return _exact_ggx(s["st"])
    return (_exact_samples(s["st"], s["q"], s["u"], case["kernel"], case["jac_eps"]), None, None,
            _exact_masking(s["st"], s["q"], s["wi"], s["wo"]))
