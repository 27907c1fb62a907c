"""The batch's one-launch sweep (Sec. 2) at the edges of its variants.

Problems join by the rows a thread of the one-CTA sweep holds (1 to 4) and by
its thread bound: planes of 31^2 (one row, 1024 threads), 24 x 22 (one, 768),
44^2 (two, 1024), 38 x 36 (two, 768), 47 x 48 (three, 768) and 600 x 4 (four,
768); 300 x 7, 52^2 (three, 1024) and 64 x 60 (four, 1024) planes sweep on
their own.  Two problems of each, in FP32 and MIXED, give the bits of the same
problems stepped alone."""
import numpy as np
import pytest

from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

# (nx, ny, nz), whether the problem joins the launch
GRIDS = [((31, 31, 4), True), ((24, 22, 5), True), ((44, 44, 4), True), ((38, 36, 4), True), ((47, 48, 4), True),
         ((600, 4, 4), True), ((300, 7, 5), False), ((52, 52, 4), False), ((64, 60, 4), False)]


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("grid, joins", GRIDS)
def test_members_keep_their_bits(grid, joins, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    spec = inputs.ragged_mixed(grid=grid, G=2, L=3)
    spec.box = tuple((n - 1) / 16.0 for n in grid)
    made = []
    for i in range(6):
        s = native.Solver.from_spec(spec, precision=precision)
        s.set_sweep_schedule(1, 1024)
        s.set_state(inputs.random_state(spec, seed=50 + i % 2))
        made.append(s)
    one, own, alone = made[:2], made[2:4], made[4:]
    b1, b0 = native.Batch(one), native.Batch(own)
    b1.set_sweep_mode(1)
    launches = []
    for b in (b1, b0):
        b.step(2)
        n = native.launch_count()
        b.step(3)
        launches.append(native.launch_count() - n)
    # a step's two sweeps in one launch
    assert launches[0] == launches[1] - (3 if joins else 0)
    for x, y, z in zip(one, own, alone):
        z.step(5)
        want = z.get_state()
        assert np.array_equal(x.get_state(), want)
        assert np.array_equal(y.get_state(), want)
    b1.close()
    b0.close()
    for s in made:
        s.close()
