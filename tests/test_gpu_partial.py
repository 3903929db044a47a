"""Partly visible triangles of the projected area one by one: a vertex or an edge
close to the visibility boundary, edges that dip into view between vertices that
do not, slivers, normals collapsed onto a segment.

The reference is quadrature in 64 bits of the part that is in view (perf/cases.py),
and the oracle too where |cross| > 1e-7: its closed form divides by |cross|, and
loses its digits below that (|cross| = 3.7e-11: 2.167e-5 where the mean over ten
million points is 2.650e-5)."""
import numpy as np
import pytest
import torch

import oracle
from perf import cases

pytestmark = pytest.mark.gpu
DEV = "cuda"
SIGMA = 0.08  # texels: 4 sigma reach one triangle's centroid alone


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


def lift(m):
    m = np.asarray(m, np.float64)
    return np.concatenate([m, np.sqrt(np.maximum(0.0, 1.0 - (m * m).sum(-1, keepdims=True)))], -1)


def unit(v):
    return v / np.maximum(np.linalg.norm(v, axis=-1, keepdims=True), 1e-300)


def values(P, tri, w):
    """V / |cross| of each triangle (count, 3, 2) at its direction (count, 3), the
    quadrature's and the oracle's: quad (2 i, 2 j) of a map holds one triangle, and a footprint
    within it takes that triangle alone."""
    count = len(tri)
    side = int(np.ceil(np.sqrt(count)))
    st = np.zeros((2 * side, 2 * side, 2), np.float32)
    i, j = 2 * (np.arange(count) % side), 2 * (np.arange(count) // side)
    st[j, i], st[j, i + 1], st[j + 1, i], st[j + 1, i + 1] = tri[:, 0], tri[:, 1], tri[:, 2], tri[:, 0]
    q = np.zeros((count, 8), np.float32)
    q[:, 0], q[:, 1], q[:, 2], q[:, 4] = i + 1 / 3, j + 1 / 3, SIGMA ** 2, SIGMA ** 2
    st, q, w = torch.from_numpy(st), torch.from_numpy(q), torch.from_numpy(np.ascontiguousarray(w, np.float32))
    h = P.pndf_build_hierarchy(st.to(DEV))
    got = P.pndf_diffuse_projected_area(h, q.to(DEV), w.to(DEV)).cpu().double().numpy()
    h.free()
    k = 2 * np.pi * SIGMA ** 2
    t = torch.from_numpy(tri).to(DEV).double()
    d = w.to(DEV).double()
    quadrature = cases._visible(t[:, 0], t[:, 1], t[:, 2], (d / d.norm(dim=1, keepdim=True)).T.contiguous())
    return got * k, quadrature.cpu().numpy(), oracle.projarea(st, q, w) * k


def visible_share(tri, w, n=48):
    """Share of each triangle's uv that sees w, by its cells' centres."""
    u = (np.arange(n) + 0.5) / n
    s, t = (v[None].repeat(len(tri), 0) for v in (np.tile(u, n), np.repeat(u, n)))
    s, t = np.where(s + t > 1, 1 - s, s), np.where(s + t > 1, 1 - t, t)
    m = tri[:, None, 0] + s[..., None] * (tri[:, None, 1] - tri[:, None, 0]) + t[..., None] * (tri[:, None, 2] - tri[:, None, 0])
    return (np.einsum("kpc,kc->kp", lift(m), np.asarray(w, np.float64)) > 0).mean(1)


def check(P, tri, w):
    """The value is half the mean of w . m~ / m~_z over the visible part, so an
    error e of w . m~ moves it by e share / (2 m~_z): FP32 directions, normals and
    products give e < 5e-7, m~_z > 0.5 here.  1e-4 relative covers the quadrature,
    1e-8 the share's own resolution."""
    tri = np.asarray(tri, np.float32)
    w = np.asarray(w, np.float32)
    got, ref, closed = values(P, tri, w)
    tol = 5e-7 * visible_share(tri.astype(np.float64), w) + 1e-8
    e = tri[:, 1:].astype(np.float64) - tri[:, :1]
    cross = np.abs(e[:, 0, 0] * e[:, 1, 1] - e[:, 0, 1] * e[:, 1, 0])
    for r in (ref, np.where(cross > 1e-7, closed, ref)):
        err = np.abs(got - r) - (1e-4 * r + tol)
        k = int(np.argmax(err))
        assert err[k] <= 0, (got[k], r[k], tri[k].tolist(), w[k].tolist(), int((err > 0).sum()))
    return ref


def test_known_triangles(P):
    tri = [[(.2263, .3805), (.1619, .4), (.3029, .1626)], [(-.4, .1329), (-.4, -.4), (-.4, .0543)],
           [(-.3516, .3567), (-.2311, .4), (.4, .4)], [(-.3, .3), (-.3, -.2), (-.3, .3)]]
    w = [(-.8283, -.4425, .3438), (.9123, -.0707, .4035), (.0043, -.9177, .3972), (.9507792, .01683164, .30941176)]
    ref = check(P, tri, w)
    assert abs(ref[1] - 3.34e-3) < 1e-5


@pytest.mark.parametrize("third", [(0.0, 0.7), (0.0, 0.52), (0.0, 0.3), (0.1, 0.6), (-0.2, 0.5)])
def test_edge_along_the_boundary(P, third):
    """Two mirrored normals at the same w . m~, from both sides of 0."""
    a, b = (-0.2, 0.5), (0.2, 0.5)
    ax = unit(np.cross(lift(a), lift(b)))
    ax = -ax if ax[2] < 0 else ax
    if ax[1] > 0:  # the visible region on the origin's side
        ax = -ax * np.sign(ax[2])
    mid = unit(lift(a) + lift(b))
    eps = np.array([s * 10.0 ** -k for k in np.arange(2, 8.1, 0.25) for s in (-1, 1)])
    w = unit(ax + eps[:, None] * mid)
    for order in ((0, 1, 2), (1, 2, 0), (2, 1, 0)):
        pts = np.array([a, b, third])[list(order)]
        check(P, np.repeat(pts[None], len(w), 0), w)


@pytest.mark.parametrize("kind", ["flakes", "grooves", "noise", "steep", "slivers", "collapsed"])
@pytest.mark.parametrize("near", ["edge", "vertex", "hemisphere"])
def test_triangles_near_the_boundary(P, kind, near):
    """Directions almost perpendicular to one normal or to two."""
    rng = np.random.default_rng(7)
    count = 20000
    c0, c1 = rng.normal(0, 0.15, (count, 1, 2)), rng.normal(0, 0.15, (count, 1, 2))
    if kind == "flakes":  # two cells meet in the triangle
        tri = np.where(rng.random((count, 3, 1)) < 0.5, c0, c1) + rng.normal(0, 0.005, (count, 3, 2))
    elif kind == "grooves":
        tri = np.where(rng.random((count, 3, 1)) < 0.5, 0.25, -0.25) * unit(c0) + rng.normal(0, 0.02, (count, 3, 2))
    elif kind == "noise":
        tri = rng.normal(0, 0.3, (count, 3, 2))
    elif kind == "steep":
        tri = 0.5 * unit(c0) + rng.normal(0, 0.1, (count, 3, 2))
    elif kind == "slivers":
        tri = c0 + rng.normal(0, 0.2, (count, 3, 1)) * unit(c1) + rng.normal(0, 0.3, (count, 3, 2)) * 10.0 ** rng.uniform(-7, -1, (count, 1, 1))
    else:
        tri = c0 + rng.choice([0.0, 0.1, 0.25, -0.3], (count, 3, 1)) * np.array([3.0, 4.0]) / 5
    tri = np.clip(tri, -0.4, 0.4).astype(np.float32)
    lifted = lift(tri)
    if near == "hemisphere":
        z, ph = rng.uniform(0.01, 0.6, count), rng.uniform(0, 2 * np.pi, count)
        w = np.stack([np.sqrt(1 - z * z) * np.cos(ph), np.sqrt(1 - z * z) * np.sin(ph), z], 1)
    else:
        w = np.cross(lifted[:, 0], lifted[:, 1]) if near == "edge" else np.zeros((count, 3))
        w = np.where(np.linalg.norm(w, axis=1, keepdims=True) > 1e-9, w, np.cross(lifted[:, 0], rng.normal(size=(count, 3))))
        w = unit(w)
        for v in (0, 1):
            w += lifted[:, v] * 10.0 ** rng.uniform(-8, -1.5, (count, 1)) * rng.choice([-1, 1], (count, 1))
        w = unit(w * np.where(w[:, 2:] < 0, -1, 1))
    w = w[w[:, 2] > 1e-3], tri[w[:, 2] > 1e-3]
    check(P, w[1], w[0])
