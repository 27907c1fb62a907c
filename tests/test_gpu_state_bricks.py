"""States copied by bricks and element by element (Sec. 2): a state large
enough for the bricks, given and taken on the device, against the same state
through the host, whose pieces are small; full, ragged and narrow planes, and
copies of a caller's stream."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("grid, G, L", [((24, 23, 22), 8, 5), ((33, 31, 12), 4, 7), ((9, 20, 40), 16, 5),
                                        ((4, 40, 40), 8, 5)])
def test_device_copies_match_host_copies(precision, grid, G, L):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    spec = inputs.ragged_mixed(grid=grid, G=G, L=L)
    I = inputs.hash_state_torch(spec, 5).view(spec.Nc, spec.G, spec.N).contiguous()
    if precision != "fp64":
        I = I.float().double()  # values a single-precision state holds
    host = I.cpu().numpy()
    s = native.Solver.from_spec(spec, precision=precision)
    st = torch.cuda.Stream()
    s.set_state_dev(I, st.cuda_stream)
    assert np.array_equal(s.get_state(), host)
    s.zero_state()
    s.set_state(host)
    out = torch.full_like(I, float("nan"))
    s.get_state_dev(out)
    torch.cuda.synchronize()
    assert torch.equal(out, I)
    s.close()
