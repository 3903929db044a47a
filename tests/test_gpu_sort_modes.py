"""The order a caller asks for is made, whatever the batch's size, and changes no
result: every sort mode on both sides of the sizes where the default leaves its
order out, with footprints divided and whole."""
import pytest
import torch

from paper_2505_08985_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
SORT_KERNELS = 3  # key, scan, place


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


@pytest.mark.parametrize("nq", [1, 2048, 8193, 20000])
@pytest.mark.parametrize("split", [True, False])
def test_every_order_is_made(P, nq, split):
    st = synth.flake_normals(300, 500, seed=5).to(DEV)
    q = synth.make_queries(st, nq, synth.QueryMix(sigma=(0.5, 40.0), frac_near=0.9), 5)
    h = P.pndf_build_hierarchy(st)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def run(**kw):
        before = P.pndf_launch_count()
        D = P.pndf_eval_batch_ex(h, q, split=split, **kw)
        return D, P.pndf_launch_count() - before

    whole, _ = run(sort=P.PNDF_SORT_NONE)
    plan = 2 if split else 0  # work and plan; split_small, one kernel, for small unsorted batches
    for mode in (P.PNDF_SORT_LEVEL_NORMAL, P.PNDF_SORT_LEVEL_TILE_NORMAL, P.PNDF_SORT_LEVEL_NORMAL_TILE):
        D, launches = run(sort=mode)
        assert launches == SORT_KERNELS + plan + 1
        assert torch.equal(D.view(torch.int32), whole.view(torch.int32))
    for shape, resident in ((dict(), 24), (dict(warps_per_cta=2, ctas_per_sm=1), 2), (dict(ctas_per_sm=1), 8)):
        D, launches = run(sort=P.PNDF_SORT_DEFAULT, **shape)
        left_out = split and nq <= 4 * resident * sms
        assert (launches < SORT_KERNELS + plan + 1) == left_out
        assert torch.equal(D.view(torch.int32), whole.view(torch.int32))
    h.free()
