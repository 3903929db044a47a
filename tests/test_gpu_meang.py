"""The projected area's triangle classes (small, large, cut by the visibility
boundary, grazed by it, closed form) against the FP64 oracle, map by map so
that each class carries the sum in some case, at the smallest maps and at
footprints from below a texel to many rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08985_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


def near_cut(q, n):
    """Requests with a triangle centroid within 1e-3 of the cut q = 16 (FP32 and
    FP64 may then differ in which triangles they sum)."""
    out = np.zeros(len(q), bool)
    for k, (x, y, sxx, sxy, syy) in enumerate(q[:, :5]):
        det = sxx * syy - sxy * sxy
        J, I = np.meshgrid(np.arange(n - 1), np.arange(n - 1), indexing="ij")
        for off in (1 / 3, 2 / 3):
            dx, dy = I + off - x, J + off - y
            qq = (syy * dx * dx - 2 * sxy * dx * dy + sxx * dy * dy) / det
            out[k] |= bool((np.abs(qq - 16.0) < 1e-3).any())
    return out


@pytest.mark.parametrize("spread", [0.002, 0.02, 0.1, 0.25, 0.45])  # normals' standard deviation
@pytest.mark.parametrize("wz", [(0.01, 0.1), (0.1, 1.0)])
@pytest.mark.parametrize("n", [2, 3, 33, 70])
def test_classes_match_oracle(P, spread, wz, n):
    """Each triangle's value is off by at most 8 roundings of g <= 1 and 1e-7 of
    quadrature error, halved and averaged with weights that sum to at most 1
    (5e-7 covers both); weights and sums are relative (2e-6)."""
    rng = np.random.default_rng(n)
    st = rng.normal(0.0, spread, (n, n, 2))
    st = np.clip(st, -0.65, 0.65).astype(np.float32)  # |m| <= 0.92
    st[: n // 2, : n // 3] = st[0, 0]                   # a plateau: collapsed normals
    st = torch.from_numpy(st)
    q = synth.make_queries(st, 120, synth.QueryMix(sigma=(0.4, max(1.0, n / 9)), aspect=(1.0, 4.0), centre_margin=-1.0), n)
    ph = rng.uniform(0, 2 * np.pi, 120)
    z = rng.uniform(*wz, 120)
    r = np.sqrt(1 - z * z)
    w = torch.from_numpy(np.stack([r * np.cos(ph), r * np.sin(ph), z], 1).astype(np.float32))
    ok = ~near_cut(q.double().numpy(), n)
    assert ok.sum() > 40
    ref = oracle.projarea(st, q, w)
    h = P.pndf_build_hierarchy(st.to(DEV))
    got = P.pndf_diffuse_projected_area(h, q.to(DEV), w.to(DEV)).cpu().double().numpy()
    h.free()
    err = np.abs(got - ref) - (5e-7 + 2e-6 * ref)
    assert err[ok].max() <= 0, (err[ok].max(), int(np.argmax(np.where(ok, err, -1))))
