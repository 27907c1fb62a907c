"""Stage a1 of the mixed path (Sec. 2.3) at every depth of its staging and
operand rings.

The depths are the largest that fit beside the resident operand, so they
follow from the angular order and from how many ordinates cross the z and y
faces first, which the node spacings decide: (3, 2) at L = 7 with 448 slots,
(4, 2) with 352 or 384, (4, 4) at L = 5; through tensor maps and,
on rows that are not 16-byte multiples, through 4-byte copies.  More items
than SMs, so that a ring runs on from one item to the next.  The projection
of a seeded state against the FP64 oracle.
"""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs
from test_gpu_parity import MIXED_TOL, _native, _oracle, rel, rel_elem

pytestmark = pytest.mark.gpu

# (nx, ny, nz), spacings, L, slots of the z- and y-class ordinates
CASES = [((12, 16, 16), (1.0, 0.8, 0.8), 7, 448),
         ((13, 16, 16), (1.0, 0.8, 0.8), 7, 448),
         ((16, 12, 12), (1.0, 1.0, 2.0), 7, 352),
         ((14, 13, 12), (1.0, 1.0, 2.0), 7, 352),
         ((12, 12, 16), (1.0, 1.2, 1.0), 7, 384),
         ((16, 12, 12), (1.0, 1.0, 1.0), 6, None),
         ((12, 16, 12), (1.0, 1.0, 1.0), 5, None)]


def _slots(spec):
    mu, _ = np.polynomial.legendre.leggauss(spec.nmu)
    phi = 2.0 * np.pi * np.arange(spec.nphi) / spec.nphi
    st = np.sqrt(1.0 - mu * mu)
    n = np.stack([st[:, None] * np.cos(phi), st[:, None] * np.sin(phi), np.repeat(mu[:, None], spec.nphi, 1)], -1)
    h = np.array([b / (m - 1) for b, m in zip(spec.box, spec.grid)])
    d = np.argmax(np.abs(n.reshape(-1, 3)) / h, axis=1)  # the axis crossed first
    return sum((int(np.sum(d == a)) + 31) // 32 * 32 for a in (1, 2))


@pytest.mark.parametrize("grid, h, L, slots", CASES)
def test_projection_at_every_depth(grid, h, L, slots):
    native = _native()
    spec = inputs.ragged_mixed(grid=grid, G=16, L=L)
    spec.box = tuple(a * (n - 1) / 16.0 for a, n in zip(h, grid))
    assert slots is None or _slots(spec) == slots
    P = _oracle(spec)
    s = native.Solver.from_spec(spec, precision="mixed")
    assert s.transform_path() == (2 if grid[0] % 4 == 0 and grid[1] % 4 == 0 else 3)
    I = inputs.random_state(spec, seed=21)
    Ish_r, J_r, H_r, K_r = P.project(I)
    for _ in range(2):
        Ish, J, H, K = s.stage_project(I)
        assert rel(Ish, Ish_r) < MIXED_TOL
        assert rel_elem(J, J_r) < MIXED_TOL
        assert rel(H, H_r) < MIXED_TOL
        assert rel(K, K_r) < MIXED_TOL
    s.close()
