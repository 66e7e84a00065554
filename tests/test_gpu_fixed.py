"""GPU tests of the FP64 contractions on the integer pipes (csrc/fixed.cuh) against the oracle.

Each line of doubles is put on the scale of its largest element, so the data here reach over that
scale: jumps by 1e4, elements that are exactly zero, magnitudes from 2^-40 to 2^40, and NaN.  The
bar is the FP64 path's, 1e-12 relative to the largest magnitude of the variable in its patch (or
cell): both sides round at 1e-16 of the terms and a step adds fewer than 1e3 of them."""
import numpy as np
import pytest

from oracle.weno import ader_weno
from paper_1406_7416_gb300 import adg, build_lib

pytestmark = pytest.mark.gpu
RTOL = 1e-12
GAMMA = 1.4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


def _patches(dim, N, count, kind, seed):
    """Patches (nvar, count, L.. x first) of subcell averages."""
    L = 2 * N + 7
    rng = np.random.default_rng(seed)
    shape = (count,) + (L,) * dim
    x = np.arange(L).reshape((1, L) + (1,) * (dim - 1))
    jump = {"smooth": 1.0, "jump": 1e4, "still": 10.0}[kind]
    side = np.broadcast_to(x < rng.integers(3, L - 3, size=(count,) + (1,) * dim), shape)
    rho = np.where(side, 1.0, 1.0 / jump) * rng.uniform(0.95, 1.05, shape)
    p = np.where(side, 1.0, 1.0 / jump) * rng.uniform(0.95, 1.05, shape)
    vel = [np.zeros(shape) if kind == "still" or k == 1 else rng.uniform(-0.2, 0.2, shape)
           for k in range(dim)]
    E = p / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return np.stack([rho] + [rho * v for v in vel] + [E])


def _update(P, dim, N, h, dt):
    import torch
    nv, count, Ns = dim + 2, P.shape[1], 2 * N + 1
    q = np.transpose(P, [1, 0] + list(range(dim + 1, 1, -1))).reshape(count, nv, -1)
    q = torch.from_numpy(np.ascontiguousarray(q)).cuda()
    v = torch.empty((count, nv, Ns ** dim), dtype=torch.float64, device="cuda")
    rc, msg = adg.subcell_update_noalloc(dim, N, GAMMA, h, dt, q.data_ptr(), count, v.data_ptr())
    assert rc == adg.OK, msg
    torch.cuda.synchronize()
    v = v.cpu().numpy().reshape((count, nv) + (Ns,) * dim)
    return np.transpose(v, [1, 0] + list(range(dim + 1, 1, -1)))


@pytest.mark.parametrize("kind", ["smooth", "jump", "still"])
@pytest.mark.parametrize("scale", [-40, 0, 40])
@pytest.mark.parametrize("dim,N,count", [(2, 1, 1), (2, 5, 7), (2, 9, 2), (3, 1, 2), (3, 3, 3)])
def test_subcell_update(dim, N, count, scale, kind):
    """The subcell predictor (with its reconstruction and fluxes) against the oracle's update."""
    P = _patches(dim, N, count, kind, seed=11 * N + dim) * 2.0 ** scale
    h = [0.01 * (1 + 0.3 * k) for k in range(dim)]
    dt = 0.1 * h[0] / dim
    ref, _ = ader_weno(P, dt, h, GAMMA, dim)
    got = _update(P, dim, N, h, dt)
    mag = np.abs(P).reshape(dim + 2, count, -1).max(axis=2).reshape((dim + 2, count) + (1,) * dim)
    mag = np.where(mag > 0, mag, mag.max(axis=0))       # a momentum that is zero: the patch's scale
    assert np.isfinite(ref).all()
    err = np.max(np.abs(got - ref) / mag)
    assert err <= RTOL, err


@pytest.mark.parametrize("dim,N", [(2, 2), (3, 1)])
def test_subcell_update_confines_nan(dim, N):
    """A patch with a NaN (and one with an infinity) leaves its neighbours in the launch alone,
    bit for bit, and does not come back finite itself."""
    h, dt = [0.01] * dim, 0.001
    P = _patches(dim, N, 5, "smooth", seed=3)
    alone = _update(P, dim, N, h, dt)
    mid = (slice(None),) + (N + 3,) * dim
    P[(0, 1) + mid[1:]] = np.nan
    P[(dim + 1, 3) + mid[1:]] = np.inf
    got = _update(P, dim, N, h, dt)
    for t in (0, 2, 4):
        np.testing.assert_array_equal(got[:, t], alone[:, t])
    for t in (1, 3):
        assert not np.isfinite(got[:, t]).all()
