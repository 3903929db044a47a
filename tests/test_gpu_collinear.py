"""Maps whose normals lie on a line: every triangle is a sliver whose cross is
rounding noise, and so is the place in uv of an FP32 hit.  The flat scan counts
hits that the pyramid prunes there; the pyramid agrees with itself, and a leaf
block that does not meet the support adds nothing."""
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


def make(n, angle, nq):
    t = torch.sin(torch.arange(n * n, dtype=torch.float32).reshape(n, n))
    st = torch.stack((0.25 * np.cos(angle) * t, 0.25 * np.sin(angle) * t), -1).float()
    mix = synth.QueryMix(sigma=(0.3, max(1.5, n / 12)), aspect=(1.0, 4.0), frac_near=1.0, near_noise=1e-7, centre_margin=-2.0)
    return st, synth.make_queries(st, nq, mix, n)


@pytest.mark.parametrize("angle", [0.4636476, 1.1, 2.0])
@pytest.mark.parametrize("n", [33, 66, 131])
def test_pyramid_agrees_with_itself(P, n, angle):
    st, q = make(n, angle, 20000)
    st, q = st.to(DEV), q.to(DEV)
    got = []
    for bounds in (P.PNDF_BOUNDS_F32, P.PNDF_BOUNDS_F16_OUTWARD):
        h = P.pndf_build_hierarchy(st, bounds_fmt=bounds)
        got += [P.pndf_eval_batch(h, q), P.pndf_eval_batch_ex(h, q, split=False), P.pndf_eval_batch_noalloc(h, q)]
        got.append(torch.cat([P.pndf_eval_batch(h, q[k:k + 4000].contiguous()) for k in range(0, 20000, 4000)]))
        h.free()
    for D in got[1:]:
        assert torch.equal(D.view(torch.int32), got[0].view(torch.int32))
    assert int((got[0] > 0).sum()) > 20


def block_qmin(q, n):
    """Least q = d^T S^-1 d over each leaf block (4 x 4 quads) of the map."""
    x, y, sxx, sxy, syy = q[:5]
    det = sxx * syy - sxy * sxy
    ia, ib, ic = syy / det, -sxy / det, sxx / det
    e = 4.0 * np.arange((n + 2) // 4)
    lo_x, lo_y = np.meshgrid(e - x, e - y, indexing="xy")
    hi_x, hi_y = lo_x + 4, lo_y + 4
    form = lambda dx, dy: ia * dx * dx + 2 * ib * dx * dy + ic * dy * dy
    best = np.full(lo_x.shape, np.inf)
    for ex in (lo_x, hi_x):
        best = np.minimum(best, form(ex, np.clip(-ib / ic * ex, lo_y, hi_y)))
    for ey in (lo_y, hi_y):
        best = np.minimum(best, form(np.clip(-ib / ia * ey, lo_x, hi_x), ey))
    return np.where((lo_x <= 0) & (hi_x >= 0) & (lo_y <= 0) & (hi_y >= 0), 0.0, best)


@pytest.mark.parametrize("kernel", ["PNDF_KERNEL_GAUSS", "PNDF_KERNEL_DISK"])
@pytest.mark.parametrize("angle", [1.1, 2.0])
def test_only_blocks_that_meet_the_support_count(P, angle, kernel):
    """Each query again on a map whose texels away from those blocks hold another
    normal: the same bits."""
    n, kern = 66, getattr(P, kernel)
    limit = 16.2 if kern == P.PNDF_KERNEL_GAUSS else 2.3  # blocks up to here stay as they are
    st, q = make(n, angle, 40000)
    h = P.pndf_build_hierarchy(st.to(DEV))
    D = P.pndf_eval_batch_ex(h, q.to(DEV), kernel=kern).cpu()
    h.free()
    at = torch.nonzero(D > 0)[:, 0][:400]
    assert len(at) > 150
    for k in at.tolist():
        meets = block_qmin(q[k].double().numpy(), n) <= limit
        keep = np.zeros((n + 4, n + 4), bool)
        for j, i in np.argwhere(meets):
            keep[4 * j:4 * j + 5, 4 * i:4 * i + 5] = True
        other = torch.where(torch.from_numpy(keep[:n, :n])[..., None], st, torch.tensor([0.6, -0.6]))
        h = P.pndf_build_hierarchy(other.to(DEV))
        got = P.pndf_eval_batch_ex(h, q[k:k + 1].to(DEV), kernel=kern).cpu()
        h.free()
        assert torch.equal(got.view(torch.int32), D[k:k + 1].view(torch.int32)), (k, got, D[k])
