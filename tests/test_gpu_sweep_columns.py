"""The column sweep where its mapping of threads to a plane is at an edge.

A thread holds R consecutive rows of a column, R the least for which the
plane's columns fit the schedule's threads.  The grids reach each variant
beyond the usual R <= 4: (63, 65, 5) planes of 65 x 63 (R = 6, a ragged last
row block), (520, 7, 4) planes of 7 x 520 (R = 8), (1100, 3, 3) planes with
more columns than threads (four column passes), (61, 47, 9) unaligned planes
whose last row block is partial.  Schedules give the same bits and each is
compared with the FP64 oracle (single precision: 2e-5, as for every schedule).

The 128^2 planes of a mixed-precision step take chi at rest from the chi0
table in the cluster sweep; chi_lab there is never written (1e-4, the mixed
path's tolerance).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


def _spec(grid, L=3):
    spec = inputs.ragged_mixed(grid=grid, G=2, L=L)
    spec.box = tuple((n - 1) / 16.0 for n in grid)  # equal spacings: every class has ordinates
    return spec


def _oracle(spec, I0):
    K, so = O.thomson_table(spec.G, spec.L)
    P = O.OracleProblem(grid=spec.grid, L=spec.L, nmu=spec.nmu, nphi=spec.nphi, edges=spec.edges,
                        alpha0=spec.alpha0, ne=spec.ne, u=spec.u, emis0=spec.emis0, K=K, sigma_out=so,
                        kappa=spec.kappa, box=spec.box)
    return P.step(I0, 1)[0]


@pytest.mark.parametrize("grid", [(63, 65, 5), (520, 7, 4), (1100, 3, 3), (61, 47, 9)])
def test_plane_shapes(native, grid):
    spec = _spec(grid)
    I0 = inputs.random_state(spec, seed=17)
    ref = _oracle(spec, I0)
    scale = np.max(np.abs(ref), axis=0, keepdims=True)
    s = native.Solver.from_spec(spec, precision="fp32")
    first, ran = None, 0
    for C, NT in [(1, 1024), (1, 512), (2, 512), (2, 1024), (4, 256)]:
        try:
            s.set_sweep_schedule(C, NT)
        except native.ShdError:
            continue
        s.set_state(I0)
        s.step(1)
        got = s.get_state()
        assert float(np.max(np.abs(got - ref) / scale)) < 2e-5, (C, NT)
        if first is None:
            first = got
        assert np.array_equal(got, first), (C, NT)
        ran += 1
    s.close()
    assert ran >= 1


def test_cluster_planes_take_chi_from_the_table(native):
    spec = _spec((128, 128, 4))
    spec.u[spec.Nc // 2:] = 0.0  # whole planes at rest
    I0 = inputs.random_state(spec, seed=18)
    ref = _oracle(spec, I0)
    s = native.Solver.from_spec(spec, precision="mixed")
    s.set_state(I0)
    s.step(1)
    got = s.get_state()
    s.close()
    assert float(np.max(np.abs(got - ref) / np.max(np.abs(ref), axis=0, keepdims=True))) < 1e-4
