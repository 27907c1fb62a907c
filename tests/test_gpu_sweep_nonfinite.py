"""A node whose source is infinite or NaN spoils the nodes downwind of it and
no others (Sec. 2): the linear sweep's interpolation reads, along an axis the
ray has no component on, the node itself, never a neighbour with weight zero
(0 * inf).  Nodes outside the bad node's domain of influence keep the bits
they have without it, in one CTA a plane and in clusters, aligned and not."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu


def _influence(spec, node):
    """[Nc][N] nodes a value at `node` can reach, by ordinate."""
    nx, ny, nz = spec.grid
    mu, _ = np.polynomial.legendre.leggauss(spec.nmu)
    phi = 2.0 * np.pi * np.arange(spec.nphi) / spec.nphi
    st = np.sqrt(1.0 - mu * mu)
    n = np.stack([st[:, None] * np.cos(phi), st[:, None] * np.sin(phi), np.repeat(mu[:, None], spec.nphi, 1)], -1)
    n = n.reshape(-1, 3)
    h = np.array([b / (m - 1) for b, m in zip(spec.box, spec.grid)])
    out = np.zeros((nz, ny, nx, len(n)), bool)
    z0, y0, x0 = node // (nx * ny), node // nx % ny, node % nx
    for k, v in enumerate(n):
        s = np.where(np.abs(v) < 1e-9, 0, np.sign(v)).astype(int)
        m = np.zeros((nz, ny, nx), bool)
        m[z0, y0, x0] = True
        d = int(np.argmax(np.abs(v) / h))  # the axis crossed first: one plane a step
        for _ in range(spec.grid[d]):
            new = m.copy()
            for dx in {0, s[0]}:
                for dy in {0, s[1]}:
                    for dz in {0, s[2]}:
                        if (dx, dy, dz)[d] == 0:
                            continue
                        sh = np.zeros_like(m)
                        src = tuple(slice(max(0, -a), min(w, w - a)) for a, w in zip((dz, dy, dx), m.shape))
                        dst = tuple(slice(max(0, a), min(w, w + a)) for a, w in zip((dz, dy, dx), m.shape))
                        sh[dst] = m[src]
                        new |= sh
            m = new
        out[..., k] = m
    return out.reshape(spec.Nc, len(n))


@pytest.mark.parametrize("grid, schedules", [((32, 32, 8), [(1, 1024), (1, 256), (2, 256), (4, 256)]),
                                             ((21, 19, 9), [(1, 1024), (1, 256)])])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_only_downwind_nodes_are_spoiled(grid, schedules, bad):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    spec = inputs.ragged_mixed(grid=grid, G=2, L=3)
    spec.box = tuple((n - 1) / 16.0 for n in grid)
    rng = np.random.Generator(np.random.PCG64(6))
    shape = (spec.Nc, spec.G, spec.N)
    I0, eta, chi = (rng.uniform(0.5, 1.5, shape) for _ in range(3))
    node = (grid[2] // 2 * grid[1] + grid[1] // 2) * grid[0] + grid[0] // 3
    reach = np.repeat(_influence(spec, node)[:, None, :], spec.G, 1)
    spoilt = eta.copy()
    spoilt[node] = bad
    s = native.Solver.from_spec(spec, precision="fp32")
    for C, NT in schedules:
        s.set_sweep_schedule(C, NT)
        want = s.stage_sweep(I0, eta, chi)
        got = s.stage_sweep(I0, spoilt, chi)
        assert not np.any(np.isfinite(got[node, :, :]) & ~(want[node] == 0.0))
        assert np.array_equal(got[~reach], want[~reach]), (C, NT)
    s.close()
