"""The MIXED transforms on planes whose rows are not 16-byte multiples (Sec. 2.3):
tiles are runs of 128 nodes in plane order.  Planes of less than a run, of
exactly one, of a run and one node, and of several with a remainder, in either
group of ordinates ((x, y) planes and (y, z) planes).  One step with flow
against the FP64 oracle."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs
from test_gpu_parity import MIXED_TOL, O, _native, _oracle, rel, rel_elem

pytestmark = pytest.mark.gpu

# (nx, ny, nz): nodes of the (x, y) and (y, z) planes
GRIDS = [(5, 4, 3),     # 20, 12
         (64, 2, 3),    # 128, 6
         (43, 3, 5),    # 129, 15
         (3, 9, 57),    # 27, 513
         (6, 8, 16),    # 48, 128
         (33, 31, 4)]   # 1023, 124


@pytest.mark.parametrize("grid", GRIDS)
def test_step_on_runs(grid):
    native = _native()
    spec = inputs.ragged_mixed(grid=grid, G=3)
    P = _oracle(spec)
    s = native.Solver.from_spec(spec, precision="mixed")
    assert s.transform_path() == 3
    I0 = inputs.random_state(spec, seed=8)
    s.set_state(I0)
    s.step(1)
    J, H, K, Ish = s.moments(with_sh=True)
    I_ref, _, _ = P.step(I0, 1)
    Ish_r, J_r, H_r, K_r = P.project(I_ref)
    assert rel_elem(J, J_r) < MIXED_TOL
    assert rel(H, H_r) < MIXED_TOL
    assert rel(Ish, Ish_r) < MIXED_TOL
    f = O.moments_to_eddington(J, K)
    assert np.max(np.abs(f - O.moments_to_eddington(J_r, K_r))) < MIXED_TOL
    s.close()
