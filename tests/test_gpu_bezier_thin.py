"""The Bezier sweep where the optical depth of a step vanishes (Sec. 2).

A static problem has no time term, so a step's depth is the matter's alone
and falls below every normal number where an absorber thins out into vacuum.
Opacities down to 1e-39 per unit length (depths whose reciprocal overflows
single precision), everywhere or as the tail of a Gaussian, with a zero and a
constant source under an isotropic inflow of 1: finite, and the FP64 oracle's
intensity.  Tolerance: as for the sweep's weights at any depth, about 10 x
2^-24 a plane (16 of them) at zero attenuation, 1e-5 of the column's largest
value; FP64, whose depths vanish below 1e-308, 1e-10 as everywhere.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5, "mixed": 1e-5}


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


def _fields(spec, profile, source, tiny):
    """(eta, chi) [c][g][k]; tiny: the smallest opacity."""
    rng = np.random.Generator(np.random.PCG64(9))
    shape = (spec.Nc, spec.G, spec.N)
    if profile == "thin":
        chi = np.exp(rng.uniform(np.log(tiny), np.log(tiny) + np.log(100.0), shape))
    else:
        nx, ny, nz = spec.grid
        z, y, x = np.meshgrid(np.linspace(-1, 1, nz), np.linspace(-1, 1, ny), np.linspace(-1, 1, nx), indexing="ij")
        r2 = (x * x + y * y + z * z).ravel() / 3.0
        chi = 20.0 * np.exp(np.log(tiny / 20.0) * r2)[:, None, None] * rng.uniform(0.5, 1.5, shape)
    return (0.0 if source == "zero" else 0.7) * chi, chi


@pytest.mark.parametrize("precision, profile, source",
                         [(p, f, s) for p in ("fp32", "mixed") for f in ("thin", "tail") for s in ("zero", "constant")]
                         + [("fp64", "thin", "zero"), ("fp64", "tail", "zero")])
def test_vanishing_depths(native, precision, profile, source):
    spec = inputs.ragged_mixed(grid=(16, 13, 12), G=2, L=3)
    spec.kappa = 0.0
    eta, chi = _fields(spec, profile, source, 1e-309 if precision == "fp64" else 1e-39)
    I0 = np.random.Generator(np.random.PCG64(10)).uniform(0.5, 1.5, chi.shape)
    if precision != "fp64":  # single-precision values on both sides
        eta, chi, I0 = (a.astype(np.float32).astype(np.float64) for a in (eta, chi, I0))
    spec.alpha0[:] = max(20.0, chi.max())
    K, so = O.thomson_table(spec.G, spec.L)
    P = O.OracleProblem(grid=spec.grid, L=spec.L, nmu=spec.nmu, nphi=spec.nphi, edges=spec.edges,
                        alpha0=spec.alpha0, ne=spec.ne, u=spec.u, emis0=spec.emis0, K=K, sigma_out=so,
                        kappa=0.0, box=spec.box)
    P.set_integrator("bezier")
    P.set_bc(1, np.ones(spec.G))
    ref = P.sweep(I0, eta, chi)
    assert np.all(np.isfinite(ref))
    s = native.Solver.from_spec(spec, precision=precision)
    s.set_integrator("bezier")
    s.set_boundary(native.BC_ISO, np.ones(spec.G))
    got = s.stage_sweep(I0, eta, chi)
    s.close()
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref) / np.max(np.abs(ref), axis=0, keepdims=True)) < TOL[precision]
