"""The position behind a sampled normal, seen through a map that rises or falls by
2 per texel along either axis: normals next to 0 show it to 1e-10 of a texel and
finer.  Against extended precision, the offset is good to 1e-12 of sigma (FP64
reaches 6e-13 with the Gaussian, where U1 is next to 0)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"
N = 4096
NEAR = 0.01  # normals looked at


@pytest.fixture(scope="module")
def P():
    from paper_2505_08985_gb300 import pndf
    return pndf


def positions(q, u, kernel):
    """x + L v in extended precision."""
    q, u = q.astype(np.longdouble), u.astype(np.longdouble)
    if kernel == 2:
        v = 1.5 * (2 * u - 1)
    else:
        # log(1 - U1 (1 - e^-8)) as log1p, which FP64 inputs next to 0 need
        rad = 1.5 * np.sqrt(u[:, 0]) if kernel == 1 else np.sqrt(-2 * np.log1p(u[:, 0] * np.expm1(np.longdouble(-8))))
        ang = 2 * np.arccos(np.longdouble(-1)) * u[:, 1]
        v = np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1)
    l11 = np.sqrt(q[:, 2])
    l21 = q[:, 3] / l11
    l22 = np.sqrt(q[:, 4] - l21 * l21)
    return np.stack([q[:, 0] + l11 * v[:, 0], q[:, 1] + l21 * v[:, 0] + l22 * v[:, 1]], 1)


@pytest.mark.parametrize("kernel", [0, 1, 2])
@pytest.mark.parametrize("where", ["uniform", "first 1e-4", "last 1e-3"])
@pytest.mark.parametrize("sigma", [3.0, 60.0, 480.0])
def test_positions(P, kernel, where, sigma):
    rng = np.random.default_rng(17)
    count = 200000
    zigzag = 1.0 - 2.0 * (np.arange(N) & 1)
    st = np.empty((N, N, 2), np.float32)
    st[..., 0], st[..., 1] = zigzag[None, :], zigzag[:, None]
    u = rng.random((count, 2), dtype=np.float32)
    if where == "first 1e-4":
        u[:, 0] *= 1e-4
    elif where == "last 1e-3":
        u[:, 0] = 1 - np.float32(1e-3) * u[:, 0]
    a, b = sigma ** 2, (sigma / rng.uniform(1, 4, count)) ** 2
    th = rng.uniform(0, np.pi, count)
    q = np.zeros((count, 8), np.float32)
    q[:, :2] = N / 2 + rng.uniform(-20, 20, (count, 2))
    q[:, 2] = a * np.cos(th) ** 2 + b * np.sin(th) ** 2
    q[:, 3] = (a - b) * np.cos(th) * np.sin(th)
    q[:, 4] = a * np.sin(th) ** 2 + b * np.cos(th) ** 2
    h = P.pndf_build_hierarchy(torch.from_numpy(st).to(DEV))
    m, tri, flags = P.pndf_sample_normals(h, torch.from_numpy(q).to(DEV), torch.from_numpy(u).to(DEV), kernel=kernel)
    h.free()
    assert int(flags.abs().sum()) == 0
    x = positions(q, u, kernel)
    i = np.floor(x)
    ref = (1 - 2 * (x - i)) * (1 - 2 * np.mod(i, 2))
    near = np.abs(ref) < NEAR
    assert near.sum() > 1000
    err = np.abs(m.cpu().numpy().astype(np.longdouble) - ref) - np.abs(ref) * 2.0 ** -23
    assert err[near].max() <= 2 * 1e-12 * sigma, float(err[near].max() / (2 * sigma))
