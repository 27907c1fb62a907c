"""The single-precision transforms (stages a1 and a3) at the edges of their
tiles, against the FP64 oracle.

Grids with runs that are and are not 16-byte multiples, an odd number of
8 x 8 bricks, one group and several; ordinate counts that are not multiples
of 4 or 16, the group of 16 in which the x-class begins, angular orders from
1 to 8 (at 8 the resident harmonics of a3 no longer fit and the tiled kernel
runs).  2e-5 of each field's scale, the single-precision tolerance of every
parity test (sums over up to 648 ordinates x 81 harmonics of values rounded
at 6e-8).  Steps: chi_lab at nodes at rest is kept from one fill, through a
change of the absorption and of the moving nodes (three steps, 3 x 2e-5).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


def _problem(spec):
    K, so = O.thomson_table(spec.G, spec.L)
    return O.OracleProblem(grid=spec.grid, L=spec.L, nmu=spec.nmu, nphi=spec.nphi, edges=spec.edges,
                           alpha0=spec.alpha0, ne=spec.ne, u=spec.u, emis0=spec.emis0, K=K, sigma_out=so,
                           kappa=spec.kappa, box=spec.box)


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("grid, G, L, mesh", [((9, 7, 5), 3, 3, None), ((8, 8, 3), 1, 3, None), ((12, 20, 3), 2, 5, None),
                                              ((6, 10, 4), 2, 7, None), ((17, 4, 3), 2, 1, (3, 5)),
                                              ((4, 12, 3), 2, 2, (5, 7)), ((7, 5, 3), 1, 8, None)])
def test_transforms(native, grid, G, L, mesh):
    spec = inputs.ragged_mixed(grid=grid, G=G, L=L)
    if mesh:
        spec.nmu, spec.nphi = mesh
    P = _problem(spec)
    I = inputs.random_state(spec, seed=5)
    Ish, J, H, K = P.project(I)
    S = P.source(Ish)
    eta, chi = P.sh2lab(S)
    s = native.Solver.from_spec(spec, precision="fp32")
    gI, gJ, gH, gK = s.stage_project(I)
    geta, gchi = s.stage_sh2lab(S)
    s.close()
    for name, a, b in (("I_lm", gI, Ish), ("J", gJ, J), ("H", gH, H), ("K", gK, K), ("eta", geta, eta), ("chi", gchi, chi)):
        assert _rel(a, b) < TOL, (name, _rel(a, b))


@pytest.mark.parametrize("grid", [(12, 12, 6), (6, 10, 4), (9, 7, 5)])
@pytest.mark.parametrize("integrator", ["linear", "bezier"])
def test_chi_at_rest_is_kept(native, grid, integrator):
    spec = inputs.ragged_mixed(grid=grid, G=3, L=3)
    spec.u[spec.Nc // 3: spec.Nc // 2] = 0.0
    I = inputs.random_state(spec, seed=6)
    s = native.Solver.from_spec(spec, precision="fp32")
    s.set_integrator(integrator)
    s.set_state(I)
    for leg in range(3):
        if leg == 1:
            spec.alpha0 = spec.alpha0 * 1.7
        if leg == 2:
            spec.u[::5] = 0.0
        if leg:
            s.set_fields(spec.alpha0, spec.ne, spec.u, spec.emis0)
        s.step(1)
        P = _problem(spec)
        P.set_integrator(integrator)
        I = P.step(I, 1)[0]
        got = s.get_state()
        err = float(np.max(np.abs(got - I) / np.max(np.abs(I), axis=0, keepdims=True)))
        assert err < 3 * TOL, (leg, err)
    s.close()
