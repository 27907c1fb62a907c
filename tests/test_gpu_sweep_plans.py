"""Every schedule that a problem accepts runs the column sweep, with the bits
of every other (Sec. 2).

The schedules accepted are listed, so that none is dropped unseen.  Grids:
planes of 584 to 1132 columns, whose halo slots are two instead of four where
four leave no room (one to eight rows a thread and four column passes);
(64, 30, 10) and (60, 44, 20), whose last CTA has
fewer rows than the others or none.  Against the oracle within 2e-5, the
tolerance of every schedule.

The 128^2 planes of a mixed-precision step take chi at rest from the chi0
table: after a caller's chi_lab of NaN no kernel fills it, as one does on
grids whose rows are not multiples of 4, and the step keeps its bits.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1507_05141_gb300 import inputs

pytestmark = pytest.mark.gpu

CANDIDATES = [(1, 1024), (1, 512), (1, 256)] + [(C, NT) for C in (2, 4, 8, 16) for NT in (256, 384, 512, 768, 1024)]
GRIDS = {
    (1000, 16, 8): [(4, 1024), (8, 512), (8, 768), (8, 1024), (16, 256), (16, 384), (16, 512), (16, 1024)],
    (780, 20, 8): [(4, 1024), (8, 1024), (16, 512), (16, 768), (16, 1024)],
    (8, 584, 28): [(4, 1024), (8, 1024), (16, 512), (16, 1024)],
    (1132, 4, 12): [(4, 1024), (8, 768), (8, 1024), (16, 384), (16, 512), (16, 1024)],
    (64, 30, 10): [(1, 1024), (1, 512), (2, 256), (2, 384), (2, 512), (2, 1024), (4, 256), (4, 512), (8, 256)],
    (60, 44, 20): [(1, 1024), (2, 512), (2, 1024), (4, 256), (4, 512), (4, 1024), (8, 256), (8, 512), (16, 256)],
}


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05141_gb300 import native
    return native


def _spec(grid, L):
    spec = inputs.ragged_mixed(grid=grid, G=1 if L == 1 else 2, L=L)
    spec.box = tuple((n - 1) / 16.0 for n in grid)  # equal spacings: every class has ordinates
    return spec


def _schedules(native, s):
    for C, NT in CANDIDATES:
        try:
            s.set_sweep_schedule(C, NT)
        except native.ShdError:
            continue
        yield C, NT


@pytest.mark.parametrize("grid", list(GRIDS))
def test_accepted_schedules_agree(native, grid):
    spec = _spec(grid, 1)
    I0 = inputs.random_state(spec, seed=27)
    K, so = O.thomson_table(spec.G, spec.L)
    ref = O.OracleProblem(grid=spec.grid, L=spec.L, nmu=spec.nmu, nphi=spec.nphi, edges=spec.edges,
                          alpha0=spec.alpha0, ne=spec.ne, u=spec.u, emis0=spec.emis0, K=K, sigma_out=so,
                          kappa=spec.kappa, box=spec.box).step(I0, 1)[0]
    scale = np.max(np.abs(ref), axis=0, keepdims=True)
    s = native.Solver.from_spec(spec, precision="fp32")
    ran, first = [], None
    for sched in _schedules(native, s):
        s.set_state(I0)
        s.step(1)
        got = s.get_state()
        assert np.max(np.abs(got - ref) / scale) < 2e-5, sched
        first = got if first is None else first
        assert np.array_equal(got, first), sched
        ran.append(sched)
    s.close()
    assert ran == GRIDS[grid]


@pytest.mark.parametrize("grid, fills", [((128, 128, 4), 0), ((126, 128, 4), 1)])
def test_chi_at_rest_is_taken_from_the_table(native, grid, fills):
    spec = _spec(grid, 3)
    spec.u[spec.Nc // 2:] = 0.0  # whole planes at rest
    I0 = inputs.random_state(spec, seed=18)
    s = native.Solver.from_spec(spec, precision="mixed")
    first, ran = None, 0
    for sched in _schedules(native, s):
        counts = []
        for spoil in (False, True):
            if spoil:
                s.stage_sweep(I0, np.ones_like(I0), np.full_like(I0, np.nan))
            else:
                s.set_state(I0)
                s.step(1)
            s.set_state(I0)
            n = native.launch_count()
            s.step(1)
            counts.append(native.launch_count() - n)
            got = s.get_state()
            first = got if first is None else first
            assert np.array_equal(got, first), sched
        assert counts[1] == counts[0] + fills, sched
        ran += 1
    s.close()
    assert ran >= 5
