"""State copies between the canonical FP64 layout and the library's.

The copies move 8 x 8 bricks of nodes x 32 ordinates: grids with partial
bricks, ordinate counts that are not multiples of 32, one group, and a host
copy larger than the staging buffer (its pieces end inside a layer of
bricks).  FP64 comes back bit for bit, single precision as its rounding.
"""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("grid, G, L, mesh", [((9, 7, 5), 3, 3, None), ((8, 16, 3), 1, 1, (3, 5)), ((17, 3, 2), 2, 2, (5, 7)),
                                              ((30, 28, 10), 8, 5, None)])
def test_round_trip(native, precision, grid, G, L, mesh):
    import torch
    spec = inputs.ragged_mixed(grid=grid, G=G, L=L)
    if mesh:
        spec.nmu, spec.nphi = mesh
    I = inputs.random_state(spec, seed=8)
    want = I if precision == "fp64" else I.astype(np.float32).astype(np.float64)
    s = native.Solver.from_spec(spec, precision=precision)
    s.set_state(I)
    assert np.array_equal(s.get_state(), want)
    dev = torch.zeros(spec.Nc, spec.G, spec.N, dtype=torch.float64, device="cuda")
    s.get_state_dev(dev)
    assert np.array_equal(dev.cpu().numpy(), want)
    s.zero_state()
    s.set_state_dev(torch.from_numpy(I).cuda())
    assert np.array_equal(s.get_state(), want)
    s.close()
