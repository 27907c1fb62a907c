"""The moments of one state are one set of values: J, H, K of moments(), of
moments(with_sh=True), of moments_dev and of project_noalloc agree bit for bit
in every precision and on every transform path (tensor maps, ragged rows, CUDA
cores), and so do the comoving projections."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("grid", [(16, 12, 8), (9, 7, 6)])
def test_every_call_gives_the_same_moments(precision, grid):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    spec = inputs.ragged_mixed(grid=grid, G=3)
    s = native.Solver.from_spec(spec, precision=precision)
    s.set_state(inputs.random_state(spec, seed=23))
    s.step(2)
    plain = s.moments()
    *with_sh, Ish = s.moments(with_sh=True)
    dev = torch.empty(s.Nc, s.G, 10, dtype=torch.float64, device="cuda")
    s.moments_dev(dev)
    torch.cuda.synchronize()
    for a, b in zip(plain, with_sh):
        assert np.array_equal(a, b)
    assert np.array_equal(dev.cpu().numpy(), np.concatenate([plain[0][..., None], plain[1], plain[2]], -1))
    dt = torch.float64 if precision == "fp64" else torch.float32
    Ish_n, mom_n = torch.empty(Ish.shape, dtype=dt, device="cuda"), torch.empty(dev.shape, dtype=dt, device="cuda")
    s.project_noalloc(Ish_n, mom_n)
    torch.cuda.synchronize()
    assert torch.equal(mom_n.double(), dev)
    assert np.array_equal(Ish_n.double().cpu().numpy(), Ish)
    assert np.array_equal(Ish, s.stage_project(s.get_state())[0])
    s.close()
