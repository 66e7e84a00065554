"""GPU: options set on a state while it is in a batch.  Some options are read on the device from the
state's parameters, others choose the launches of its group; from the batch's next step on both are
the new ones, so the state ends bit for bit where the same options take it alone."""
import numpy as np
import pytest

from paper_1406_7416_gb300 import adg, build_lib, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


CASES = {
    # split traces become FP64 ones on a periodic axis (block-per-cell and warp-per-cell shapes)
    "fp64_sweep_N6": (6, adg.PREC_MIXED_FP32, [(adg.OPT_FP64_SWEEPS, 0)], [(adg.OPT_FP64_SWEEPS, 1)]),
    "split_N6": (6, adg.PREC_MIXED_FP32, [], [(adg.OPT_FP64_SWEEPS, 0)]),
    "fp64_sweep_N3": (3, adg.PREC_MIXED_FP32, [], [(adg.OPT_FP64_SWEEPS, 2)]),
    "fp64_sweep_block": (2, adg.PREC_MIXED_FP32, [(adg.OPT_PREDICTOR, adg.PRED_BLOCK)],
                         [(adg.OPT_FP64_SWEEPS, 1)]),
    "flux_fp64": (3, adg.PREC_FP64, [], [(adg.OPT_FLUX, adg.FLUX_OSHER)]),
    "flux_mixed": (3, adg.PREC_MIXED_FP32, [], [(adg.OPT_FLUX, adg.FLUX_OSHER)]),
    "subcell_fp64": (3, adg.PREC_MIXED_FP32, [],
                     [(adg.OPT_SUBCELL_FP32, 0), (adg.OPT_SUBCELL_FP64_SWEEPS, 3)]),
    "no_cascade": (3, adg.PREC_FP64, [], [(adg.OPT_CASCADE, 0)]),
    "iterations": (2, adg.PREC_MIXED_FP32, [], [(adg.OPT_PICARD_ITERS, 1)]),
}


@pytest.mark.parametrize("fixed_dt", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_options_of_a_batched_state(name, fixed_dt):
    N, prec, before, after = CASES[name]
    w = inputs.quadrants_vortex_2d(n=8, N=N)
    cfl = 0.5 * w["cfl"]

    def make():
        s = adg.Solver.from_workload(w, prec)
        for key, value in before:
            s.set_option(key, value)
        s.init_problem(w["problem"])
        return s

    alone, still, member, other = (make() for _ in range(4))
    dt = alone.max_dt(cfl)
    batch = adg.Batch([member, other])

    def steps(count):
        for _ in range(count):
            for s in (alone, still):
                s.step(dt) if fixed_dt else s.step_cfl(cfl)
            batch.step(np.array([dt, dt])) if fixed_dt else batch.step(cfl=cfl)

    steps(2)
    for key, value in after:
        member.set_option(key, value)
        alone.set_option(key, value)
    steps(3)
    batch.close()
    for a, b in ((alone, member), (still, other)):
        assert a.status() == adg.OK and b.status() == adg.OK
        for x, y in zip(a.read_full(), b.read_full()):
            np.testing.assert_array_equal(x, y)
    if name != "no_cascade":            # (no cell of this flow needs the first-order layer)
        assert not np.array_equal(member.read(), other.read())
    for s in (alone, still, member, other):
        s.close()
