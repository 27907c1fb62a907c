"""FP64 problems near the device's memory limit.

The remap tables of moving nodes only save time, so they never take memory a
problem needs: with little left free the remaps compute in place, and tables
held when an allocation of the library's fails are given back for it.  The
free memory is bounded by one large allocation of the caller's; the steps give
the same bits as without it.
"""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _solver(native, spec, I0):
    s = native.Solver.from_spec(spec, precision="fp64")
    s.set_state(I0)
    return s


def _leave(torch, nbytes):
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("held", [False, True])
def test_runge_kutta_fits_beside_the_tables(held):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    spec = inputs.ragged_mixed(grid=(28, 26, 24), G=2, L=3)
    I0 = inputs.random_state(spec, seed=31)
    tables = 96 * int(np.sum(np.any(spec.u != 0, axis=1))) * spec.N
    arrays = 3 * 8 * spec.Nc * spec.N * spec.G  # what the Runge-Kutta scheme keeps
    assert tables > arrays // 2 > 48 * MB

    ref = _solver(native, spec, I0)
    plain = ref.device_bytes()
    ref.step(1)
    assert ref.device_bytes() >= plain + tables  # plenty free: the tables are taken
    ref.set_time_scheme("rk4")
    ref.step(2)
    want = ref.get_state()
    ref.close()

    s = _solver(native, spec, I0)
    fill = None
    try:
        if held:
            s.step(1)
            fill = _leave(torch, arrays - 32 * MB)
        else:
            fill = _leave(torch, arrays + tables // 2)  # not both
            s.step(1)
        s.set_time_scheme("rk4")
        s.step(2)
        got = s.get_state()
        assert s.device_bytes() < plain + arrays + tables
    finally:
        del fill
        torch.cuda.empty_cache()
        s.close()
    assert np.array_equal(got, want)
