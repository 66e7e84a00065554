"""GPU: forms of one kernel chosen by size or by boundary give the same bits.

The thread-per-node 2D predictor (several cells to a block, the last block of a cell count that is
no multiple of it, the whole sweep in registers) against the warp-per-cell one, and the face flux of
a launch with few nodes (n lanes to a node) or only interior ones (the lean form) against the same
state in a launch with a large state of other boundaries."""
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


def _predicted(N, ncell, iters, shape):
    w = inputs.quadrants_2d(n=8, N=N)
    w["ncell"], w["dx"] = ncell, (1.0 / ncell[0], 1.0 / ncell[1])
    s = adg.Solver.from_workload(w, adg.PREC_MIXED_FP32)
    s.set_option(adg.OPT_PREDICTOR, shape)
    if iters:
        s.set_option(adg.OPT_PICARD_ITERS, iters)
    s.init_problem(w["problem"])
    dt = s.max_dt(0.25 * w["cfl"])
    for _ in range(3):
        s.step(dt)
    assert s.info()["predictor"] == shape
    out = s.read_full()
    s.close()
    return out


@pytest.mark.parametrize("iters", [0, 1, 2])
@pytest.mark.parametrize("ncell", [(1, 1), (3, 7), (13, 11)])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_node_predictor_is_bitwise_the_warp_one(N, ncell, iters):
    _same(_predicted(N, ncell, iters, adg.PRED_WARP2), _predicted(N, ncell, iters, adg.PRED_WARP4))


@pytest.mark.parametrize("prec", [adg.PREC_FP64, adg.PREC_MIXED_FP32])
@pytest.mark.parametrize("name", ["periodic_2d", "open_2d", "box_2d", "box_3d"])
def test_face_flux_forms_are_bitwise_equal(name, prec):
    make = {"periodic_2d": lambda: inputs.quadrants_vortex_2d(n=7, N=3),
            "open_2d": lambda: inputs.explosion_2d(n=5, N=6),
            "box_2d": lambda: inputs.closed_box(n=6, N=1, dim=2),
            "box_3d": lambda: inputs.closed_box(n=3, N=2, dim=3)}[name]
    w = make()
    N, dim = w["N"], len(w["ncell"])
    # more node-times than one thread per lane of the chip takes: the one-thread-per-node form
    big = inputs.explosion_2d(n=100, N=N) if dim == 2 else inputs.explosion_3d(n=12, N=N)
    faces = (big["ncell"][0] + 1) * big["ncell"][0] ** (dim - 1)
    assert faces * (N + 1) ** dim > 152 * 256
    alone, mixed, other = (adg.Solver.from_workload(x, prec) for x in (w, w, big))
    for s, x in ((alone, w), (mixed, w), (other, big)):
        s.init_problem(x["problem"])
    dts = np.array([0.25 * s.max_dt(x["cfl"]) for s, x in ((mixed, w), (other, big))])
    for _ in range(2):
        alone.step(dts[0])
    batch = adg.Batch([mixed, other])
    for _ in range(2):
        batch.step(dts)
    batch.close()
    _same(alone.read_full(), mixed.read_full())
    for s in (alone, mixed, other):
        s.close()
