"""GPU: the parts of a kernel's loop that small grids do not reach, bit for bit against another form:
the thread-per-node predictor's second group of cells per block, cells of one block that take
different numbers of sweeps or none, and limiter passes that hold some of a cell's troubled
neighbours but not all."""
import numpy as np
import pytest

from paper_1406_7416_gb300 import adg, build_lib, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


def _same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


def _quadrants(ncell, N):
    w = inputs.quadrants_2d(n=8, N=N)
    w["ncell"], w["dx"] = ncell, (1.0 / ncell[0], 1.0 / ncell[1])
    return w


# more cells than the blocks of a full chip take at once (at 64 registers per thread or more)
@pytest.mark.parametrize("N,ncell", [(1, (261, 251)), (2, (181, 179)), (3, (121, 113)), (4, (91, 89)),
                                     (5, (91, 89))])
def test_node_predictor_loops(N, ncell):
    out = []
    for shape in (adg.PRED_WARP2, adg.PRED_WARP4):
        w = _quadrants(ncell, N)
        s = adg.Solver.from_workload(w, adg.PREC_MIXED_FP32)
        s.set_option(adg.OPT_PREDICTOR, shape)
        s.init_problem(w["problem"])
        dt = s.max_dt(0.25 * w["cfl"])
        for _ in range(2):
            s.step(dt)
        out.append(s.read_full())
        s.close()
    _same(*out)


@pytest.mark.parametrize("N", [1, 3, 5])
def test_node_predictor_mixes_states(N):
    """One block's cells from states of different sweep counts, one of them past its end time."""
    out = []
    for shape in (adg.PRED_WARP2, adg.PRED_WARP4):
        states = []
        for i, iters in enumerate((N + 1, 1, 2, N + 1)):
            w = _quadrants((3, 1 + 2 * i), N)
            s = adg.Solver.from_workload(w, adg.PREC_MIXED_FP32)
            s.set_option(adg.OPT_PREDICTOR, shape)
            s.set_option(adg.OPT_PICARD_ITERS, iters)
            if i == 2:
                s.set_option(adg.OPT_END_TIME, 1e-6)
            s.init_problem(w["problem"])
            states.append(s)
        batch = adg.Batch(states)
        for _ in range(4):
            batch.step(cfl=0.02)
        batch.close()
        assert states[2].time()[1] < 4 and states[0].time()[1] == 4
        out.append([x for s in states for x in s.read_full()])
        for s in states:
            s.close()
    _same(*out)


def _ghost_run(make, prec, scratch):
    w = make()
    s = adg.Solver.from_workload(w, prec)
    if scratch:
        s.set_option(adg.OPT_SCRATCH_BYTES, scratch)
    s.set_option(adg.OPT_FORCE_LIMITER, 1)
    s.init_problem(w["problem"])
    chunk = s.info()["chunk"]
    dt = s.max_dt(0.5 * w["cfl"])
    for _ in range(3):
        s.step(dt)
    out = s.read_full()
    s.close()
    return chunk, out


@pytest.mark.parametrize("prec", [adg.PREC_FP64, adg.PREC_MIXED_FP32])
@pytest.mark.parametrize("name", ["periodic", "box", "box3d"])
def test_shared_ghosts_in_short_passes(name, prec):
    """Passes of three and seven cells of grids that neither divides."""
    make = {"periodic": lambda: inputs.quadrants_2d(n=5, N=2), "box": lambda: inputs.closed_box(n=5, N=3, dim=2),
            "box3d": lambda: inputs.closed_box(n=3, N=1, dim=3)}[name]
    _, alone = _ghost_run(make, prec, 1)
    found = set()
    lo, hi = 1, 1 << 24
    budgets = np.unique(np.geomspace(lo, hi, 160).astype(np.int64))
    for budget in budgets:
        w = make()
        s = adg.Solver.from_workload(w, prec)
        s.set_option(adg.OPT_SCRATCH_BYTES, int(budget))
        s.init_problem(w["problem"])
        chunk = s.info()["chunk"]
        s.close()
        if chunk in (3, 7) and chunk not in found:
            found.add(chunk)
            _, out = _ghost_run(make, prec, int(budget))
            _same(alone, out)
    assert found == {3, 7}
