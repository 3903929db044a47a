"""Samples from triangles whose normals are infinite, not a number or next to the
largest finite number: what the weighted sum gives in 64 bits."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("jac_eps", [0.0, 1e-6])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38, -3e38])
def test_texels(value, jac_eps):
    from paper_2505_08985_gb300 import pndf
    n, nq = 33, 4000
    rng = np.random.default_rng(2)
    st = rng.normal(0, 0.1, (n, n, 2)).astype(np.float32)
    st[4::5, 2::5, 0] = value
    q = np.zeros((nq, 8), np.float32)
    q[:, :2] = rng.integers(3, n - 4, (nq, 2))
    q[:, 2] = q[:, 4] = 0.25
    u = rng.random((nq, 2), dtype=np.float32)  # box: x + 1.5 sigma (2 u - 1), exact in FP64
    h = pndf.pndf_build_hierarchy(torch.from_numpy(st).to(DEV))
    m, tri, flags = pndf.pndf_sample_normals(h, torch.from_numpy(q).to(DEV), torch.from_numpy(u).to(DEV),
                                             kernel=pndf.PNDF_KERNEL_BOX, jac_eps=jac_eps)
    h.free()
    assert int(flags.abs().sum()) == 0
    x = q[:, :2].astype(np.float64) + 0.75 * (2 * u.astype(np.float64) - 1)
    i = np.floor(x).astype(int)
    f = x - i
    up = f.sum(1) >= 1.0
    assert np.array_equal(tri.cpu().numpy() & 1, up.astype(int))
    wide = st.astype(np.float64)
    o = up.astype(int)
    a, b, c = (wide[i[:, 1] + dy, i[:, 0] + dx] for dx, dy in ((o, o), (1 - o, o), (o, 1 - o)))
    l0 = np.where(up, f.sum(1) - 1, 1 - f.sum(1))[:, None]
    lb, lc = (np.where(up, 1 - f[:, k], f[:, k])[:, None] for k in (0, 1))
    with np.errstate(all="ignore"):
        ref = l0 * a + lb * b + lc * c
        cross = np.abs((b - a)[:, 0] * (c - a)[:, 1] - (b - a)[:, 1] * (c - a)[:, 0])
        ref = ref.astype(np.float32)
    plain = ~(cross < max(jac_eps, 0.0)) if jac_eps else np.ones(nq, bool)
    got = m.cpu().numpy()
    odd = ~np.isfinite(ref) | (np.abs(ref) > 1e30)
    assert odd[plain].sum() > 200
    assert np.array_equal(np.isnan(got)[plain], np.isnan(ref)[plain])
    at = plain[:, None] & ~np.isnan(ref)
    assert np.array_equal(np.isinf(got)[at], np.isinf(ref)[at])
    at &= np.isfinite(ref)
    assert np.allclose(got[at], ref[at], rtol=3e-7, atol=3e-8)
