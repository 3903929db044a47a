"""The pruning tests of the pyramid (binary16 boxes, slabs, group edge
functions) only prune: hit sets and densities equal the flat scan's, which
tests every triangle of the footprint, at the map sizes where the layout has
edges (groups of 2 x 2 quads, leaf blocks of 4 x 4, build tiles of 64 x 64) and
on maps whose normals make the filters degenerate."""
import numpy as np
import pytest
import torch

from paper_2505_08985_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


def make_map(kind, n):
    if kind == "flake":
        return synth.flake_normals(n, max(4, n * n // 90), seed=n)
    if kind == "bumps":
        return synth.bumps_map(n=n, n_bumps=max(1, n // 8), seed=n)
    if kind == "plateaus":  # few distinct normals: repeated vertices, m on vertices
        return synth.flake_normals(n, max(4, n * n // 30), seed=n).round(decimals=2)
    return 2.0 ** -17 * synth.bumps_map(n=n, n_bumps=max(1, n // 8), seed=n)  # near-singular triangles


@pytest.mark.parametrize("kind", ["flake", "bumps", "plateaus", "minute"])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 9, 33, 64, 65, 66, 131])
def test_hierarchy_hits_what_the_flat_scan_hits(P, kind, n):
    st = make_map(kind, n)
    rng = np.random.default_rng(n)
    nq = 1200
    near = 2e-7 if kind == "minute" else 0.02
    q = synth.make_queries(st, nq, synth.QueryMix(sigma=(0.6, max(1.5, n / 6)), aspect=(1.0, 4.0), frac_near=0.9,
                                                  near_noise=near, centre_margin=-2.0), n)
    i, j = rng.integers(0, n - 1, nq // 2), rng.integers(0, n - 1, nq // 2)
    a, b = st[j, i], st[j + rng.integers(0, 2, nq // 2), i + rng.integers(0, 2, nq // 2)]
    q[:nq // 2, 5:7] = torch.where(torch.from_numpy(rng.random(nq // 2) < 0.5)[:, None], a, 0.5 * (a + b))
    q = q.to(DEV)
    cols = [P.STATS_NAMES.index(c) for c in ("hits", "hit_hash")]
    for texels in (st.to(DEV), st.to(DEV).half()):
        got = []
        for bounds in (P.PNDF_BOUNDS_F32, P.PNDF_BOUNDS_F16_OUTWARD):
            h = P.pndf_build_hierarchy(texels, bounds_fmt=bounds)
            for mode in (P.PNDF_MODE_HIERARCHY, P.PNDF_MODE_FLAT):
                s = torch.zeros(nq, P.STATS_FIELDS, dtype=torch.int32, device=DEV)
                got.append((P.pndf_eval_batch_ex(h, q, stats=s, mode=mode), s[:, cols]))
            h.free()
        for D, s in got[1:]:
            assert torch.equal(s, got[0][1]) and torch.equal(D.view(torch.int32), got[0][0].view(torch.int32))
    if kind in ("flake", "bumps", "minute"):
        assert int((got[0][1][:, 0] > 0).sum()) > 0


def test_cut_and_exact_agree_where_nothing_is_cut(P):
    """tau so small that no node is cut: the cut's own descent (slabs at the
    leaf level only) hits what the exact one hits."""
    st = synth.flake_normals(131, 200, seed=3).to(DEV)
    q = synth.make_queries(st, 2000, synth.QueryMix(sigma=(0.6, 25.0), frac_near=0.9, centre_margin=-2.0), 3)
    for bounds in (P.PNDF_BOUNDS_F32, P.PNDF_BOUNDS_F16_OUTWARD):
        h = P.pndf_build_hierarchy(st, bounds_fmt=bounds, clusters=True)
        D = P.pndf_eval_batch_ex(h, q)
        Dt = P.pndf_eval_batch_ex(h, q, tau=1e-30)
        h.free()
        assert torch.equal(D.view(torch.int32), Dt.view(torch.int32)) and int((D > 0).sum()) > 500
