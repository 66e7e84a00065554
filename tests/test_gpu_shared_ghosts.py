"""GPU test of the limiter's shared ghost subcells: a troubled cell takes the predictor of its face
ghosts from the troubled neighbour that owns them when both are in one limiter pass.  With a
scratch budget of one cell per pass nothing is shared, so both must give the same bits, over the
boundary kinds that fix a ghost's value (periodic, also where an axis wraps on itself; transmissive;
walls; inflow and moving fronts, across a periodic axis too), both dimensions and precisions."""
import numpy as np
import pytest

from paper_1406_7416_gb300 import adg, build_lib, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


def _front_periodic():
    """Fronts on the y faces moving along a periodic x axis."""
    w = inputs.quadrants_2d(n=6, N=2)
    q = [inputs.conserved_state(1.0, (0.3, 0.0), 1.0), inputs.conserved_state(0.4, (0.0, 0.1), 0.5)]
    w["bc"] = (inputs.PERIODIC, inputs.PERIODIC, inputs.FRONT, inputs.FRONT)
    w["bc_fronts"] = {f: dict(axis=0, a=-0.45, b=1.0, before=(inputs.INFLOW, q[0]),
                              after=(inputs.INFLOW, q[1])) for f in (2, 3)}
    return w


def _strip():
    """One cell along y, two along x: cells that neighbour themselves and each other twice."""
    w = inputs.quadrants_2d(n=2, N=4)
    w["ncell"], w["dx"] = (2, 1), (0.5, 1.0)
    return w


CASES = {"periodic2d_N5": lambda: inputs.quadrants_2d(n=5, N=5),
         "periodic2d_N1": lambda: inputs.quadrants_2d(n=9, N=1),
         "transmissive2d_N9": lambda: inputs.explosion_2d(n=4, N=9),
         "box2d_N3": lambda: inputs.closed_box(n=7, N=3, dim=2),
         "double_mach_N2": lambda: inputs.double_mach(nx=14, ny=4, N=2),
         "front_periodic": _front_periodic,
         "strip": _strip,
         "box3d_N1": lambda: inputs.closed_box(n=4, N=1, dim=3),
         "explosion3d_N3": lambda: inputs.explosion_3d(n=4, N=3)}


@pytest.mark.parametrize("prec", [adg.PREC_FP64, adg.PREC_MIXED_FP32])
@pytest.mark.parametrize("force", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_shared_ghosts_are_bitwise_the_computed_ones(name, force, prec):
    states = []
    for scratch in (None, 1):
        w = CASES[name]()
        s = adg.Solver.from_workload(w, prec)
        if scratch:
            s.set_option(adg.OPT_SCRATCH_BYTES, scratch)
        s.set_option(adg.OPT_FORCE_LIMITER, force)
        s.init_problem(w["problem"])
        dt = s.max_dt(0.5 * w["cfl"])
        for _ in range(3):
            s.step(dt)
        assert s.troubled_count() > 0 and (not scratch or s.info()["chunk"] == 1)
        states.append(s.read_full())
        s.close()
    for a, b in zip(*states):
        np.testing.assert_array_equal(a, b)
