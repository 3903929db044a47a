"""Batch sizes at which a call changes its launches (one-CTA plans, unsorted
batches, one-CTA band scans): every size gives each request the value it has
in any other batch."""
import pytest
import torch

from paper_2505_08985_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


@pytest.mark.parametrize("nq", [1, 1023, 1025, 8192, 8193, 14592, 14593])
def test_densities_do_not_depend_on_the_batch_size(P, nq):
    st = synth.flake_normals(512, 900, seed=8).to(DEV)
    sigma = torch.full((1,), 60.0)
    q = synth.make_queries(st, 14593, synth.QueryMix(sigma=(0.5, 6.0), frac_near=0.9), 8)
    q[::997, 2] = q[::997, 4] = sigma.item() ** 2  # a few footprints to divide
    q[::997, 3] = 0.0
    h = P.pndf_build_hierarchy(st)
    want = P.pndf_eval_batch_noalloc(h, q)  # sorted, one warp per query
    fl = torch.zeros(nq, dtype=torch.int32, device=DEV)
    part = q[14593 - nq:].contiguous()
    got = P.pndf_eval_batch(h, part, flags=fl)
    plain = P.pndf_eval_batch_ex(h, part, sort=0, split=False)
    h.free()
    assert torch.equal(got, want[14593 - nq:]) and torch.equal(got, plain) and int(fl.sum()) == 0


@pytest.mark.parametrize("nq", [1, 1024, 1025, 4096, 4097])
def test_areas_do_not_depend_on_the_batch_size(P, nq):
    st = synth.flake_normals(256, 200, seed=9).to(DEV)
    q = synth.make_queries(st, 4097, synth.QueryMix(sigma=(0.5, 3.0)), 9)
    q[7, 2] = -1.0  # invalid: NaN
    w = synth.hemisphere_dirs(4097, 9, DEV)
    h = P.pndf_build_hierarchy(st)
    want = P.pndf_diffuse_projected_area(h, q, w)
    got = P.pndf_diffuse_projected_area(h, q[:nq].contiguous(), w[:nq].contiguous())
    h.free()
    assert torch.equal(got.view(torch.int32), want[:nq].view(torch.int32))
    assert nq <= 7 or bool(got[7].isnan())
    assert P.pndf_device_status() == P.PNDF_QF_INVALID  # (cleared for whoever runs next)
