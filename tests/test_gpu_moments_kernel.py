"""The moments J, H, K of the current state in single precision (Sec. 2), the
sums over the ordinates by their own kernel, against the same sums in FP64 of
the state read back: grids at the edges of its 16 x 16 node tiles, rows with
and without 16-byte alignment, one and several energy groups, and more
ordinates than its shared memory holds coefficients for."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [  # (nx, ny, nz), G, L, (nmu, nphi)
    ((16, 16, 3), 1, 3, None),
    ((17, 16, 4), 3, 3, None),
    ((16, 18, 3), 2, 3, None),
    ((32, 20, 5), 4, 5, None),
    ((36, 12, 4), 2, 7, None),
    ((33, 31, 3), 2, 7, None),
    ((5, 4, 6), 5, 1, None),
    ((8, 20, 3), 1, 3, (18, 60)),  # 1080 ordinates
]


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s[0])) + f"_G{s[1]}_L{s[2]}")
def test_moments_are_the_quadrature(precision, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    grid, G, L, angles = shape
    spec = inputs.ragged_mixed(grid=grid, G=G, L=L, seed=3)
    if angles:
        spec.nmu, spec.nphi = angles
    s = native.Solver.from_spec(spec, precision=precision)
    s.set_state(inputs.random_state(spec, seed=5))
    I = s.get_state()
    J, H, K = s.moments()
    got = np.concatenate([J[..., None], H, K], -1)
    dev = torch.full((s.Nc, s.G, 10), float("nan"), dtype=torch.float64, device="cuda")
    s.moments_dev(dev)
    torch.cuda.synchronize()
    assert np.array_equal(dev.cpu().numpy(), got)
    s.close()

    mu, w = np.polynomial.legendre.leggauss(spec.nmu)
    phi = 2.0 * np.pi * np.arange(spec.nphi) / spec.nphi
    st = np.sqrt(1.0 - mu * mu)
    n = np.stack([st[:, None] * np.cos(phi), st[:, None] * np.sin(phi), np.repeat(mu[:, None], spec.nphi, 1)], -1)
    n = n.reshape(-1, 3)
    W = np.repeat(w * 2.0 * np.pi / spec.nphi, spec.nphi) / (4.0 * np.pi)
    f = np.stack([np.ones(len(n)), *n.T, n[:, 0] ** 2, n[:, 1] ** 2, n[:, 2] ** 2, n[:, 0] * n[:, 1],
                  n[:, 0] * n[:, 2], n[:, 1] * n[:, 2]], 1) * W[:, None]
    want = I @ f
    # each sum: chains of at most N products and additions, with coefficients rounded once
    bound = (len(n) + 10) * 2.0 ** -24 * (np.abs(I) @ np.abs(f)) + 1e-15 * np.abs(I).max()
    assert np.all(np.abs(got - want) <= bound)
