"""Sampling in pairs of FP32 numbers: the triangle and the normal of the FP64
oracle at the edges of its range (uniforms 0 and 1, whole quarter turns, variances
and centres next to the limits past which a record takes the FP64 form), and
through the FP64 form beyond them."""
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


@pytest.mark.parametrize("kernel", [0, 1, 2])
@pytest.mark.parametrize("sigma", [1.01e-4, 0.9e-4, 0.7, 90.0])
@pytest.mark.parametrize("corr", [0.0, 0.9, 0.9994, 0.9996])
def test_pairs_match_oracle(P, kernel, sigma, corr):
    """Normals agree to half an ulp of binary32 at 0.5 and 1e-9 (the position's
    error times the map's slope); triangles except within 1e-9 of an edge."""
    n, nq = 150, 2000
    rng = np.random.default_rng(5)
    st = synth.flake_normals(n, 300, seed=5)
    q = torch.zeros(nq, 8)
    q[:, 0] = torch.from_numpy(rng.uniform(2, n - 3, nq))
    q[:, 1] = torch.from_numpy(rng.uniform(2, n - 3, nq))
    asp = rng.uniform(1, 3, nq)
    q[:, 2] = torch.from_numpy((sigma * asp) ** 2)
    q[:, 4] = sigma * sigma
    q[:, 3] = corr * torch.sqrt(q[:, 2] * q[:, 4])
    U = torch.from_numpy(rng.uniform(0, 1, (nq, 2)).astype(np.float32))
    U[:40, 0] = torch.tensor([0.0, 1.0, 2.0 ** -24, 1.0 - 2.0 ** -24]).repeat(10)
    U[40:80, 1] = torch.arange(40).float() % 9 / 8
    h = P.pndf_build_hierarchy(st.to(DEV))
    m, tri, fl = (t.cpu().numpy() for t in P.pndf_sample_normals(h, q.to(DEV), U.to(DEV), kernel=kernel, jac_eps=1e-6))
    h.free()
    mo, to, fo = oracle.sample(st, q, U.numpy(), kernel=kernel, jac_eps=1e-6)
    assert np.array_equal((fl & 2) != 0, (fo & oracle.F_OUTSIDE) != 0)
    same = (fo & (oracle.F_OUTSIDE | oracle.F_NEAR_EDGE)) == 0
    assert same.sum() > nq // 8
    assert np.array_equal(tri.astype(np.int64)[same], to[same])
    assert np.abs(m.astype(np.float64) - mo)[same].max() <= 2.0 ** -26 + 1e-9
