"""The single-precision transfer weights over every optical depth.

The weights of the linear and the cubic Bezier short characteristic are
taken in single precision throughout: a series below 1/2 (linear) or 2
(Bezier), closed forms above, the exponential's argument compensated where
steps can exceed 16.  Each case sweeps random fields whose step depths span
one range, thin to opaque and across the branches, against the FP64 oracle.

Tolerance: a step's weights and depth carry a few units of 2^-24 (the
exponential's argument x has relative error of about 4 such units, and
x e^-x < 0.4), the intensity is a convex mix of bounded values, and errors
are attenuated along the ray with it: about 10 x 2^-24 times the number of
planes (16) at zero attenuation, 1e-5 of the column's largest value.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


@pytest.mark.parametrize("integrator", ["linear", "bezier"])
@pytest.mark.parametrize("lo, hi", [(1e-4, 1e-2), (0.2, 1.2), (1.0, 4.0), (12.0, 24.0), (60.0, 400.0), (1e-3, 300.0)])
@pytest.mark.parametrize("kappa", [0.0, 3.0])
def test_step_depths(native, integrator, lo, hi, kappa):
    spec = inputs.ragged_mixed(grid=(16, 13, 12), G=2, L=3)
    spec.kappa = kappa
    rng = np.random.Generator(np.random.PCG64(5))
    shape = (spec.Nc, spec.G, spec.N)
    h = 1.0 / 15.0
    chi = np.exp(rng.uniform(np.log(lo), np.log(hi), shape)) / h
    # float32 values on both sides: the sweep alone is compared
    chi = chi.astype(np.float32).astype(np.float64)
    eta = (chi * rng.uniform(0.5, 1.5, shape)).astype(np.float32).astype(np.float64)
    I0 = rng.uniform(0.5, 1.5, shape).astype(np.float32).astype(np.float64)
    # the fields bound the depths the sweep must allow for
    spec.alpha0[:] = hi / h
    K, so = O.thomson_table(spec.G, spec.L)
    P = O.OracleProblem(grid=spec.grid, L=spec.L, nmu=spec.nmu, nphi=spec.nphi, edges=spec.edges,
                        alpha0=spec.alpha0, ne=spec.ne, u=spec.u, emis0=spec.emis0, K=K, sigma_out=so,
                        kappa=spec.kappa, box=spec.box)
    P.set_integrator(integrator)
    ref = P.sweep(I0, eta, chi)
    s = native.Solver.from_spec(spec, precision="fp32", scattering="thomson")
    s.set_integrator(integrator)
    got = s.stage_sweep(I0, eta, chi)
    s.close()
    scale = np.max(np.abs(ref), axis=0, keepdims=True)
    err = float(np.max(np.abs(got - ref) / scale))
    assert err < TOL, err
