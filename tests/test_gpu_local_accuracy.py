"""GPU: FP64 results at their own scale.  The contractions on the integer pipes hold a line's
elements on the scale of its largest; beside large neighbours the small values must keep their own
last places.  Errors against the oracle are measured relative to the largest magnitude nearby (a
cell or subcell and those that touch it, whose fluxes enter it), not to that of the whole grid."""
import numpy as np
import pytest

from oracle import euler
from oracle.dg import Grid
from oracle.step import Scheme, State, stable_dt, step
from oracle.weno import ader_weno
from paper_1406_7416_gb300 import adg, build_lib

from helpers import beta_from_abi, from_abi, load_state

pytestmark = pytest.mark.gpu
RTOL = 1e-12
GAMMA = 1.4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


def _nearby(A, axes):
    """Largest magnitude over the 3^d block around each entry (periodic)."""
    A = np.abs(A)
    for ax in axes:
        A = np.maximum(A, np.maximum(np.roll(A, 1, ax), np.roll(A, -1, ax)))
    return A


@pytest.mark.parametrize("jump", [1e2, 1e4, 1e6])
@pytest.mark.parametrize("dim,N,count", [(2, 2, 6), (2, 5, 4), (3, 1, 2), (3, 2, 1)])
def test_subcell_update_beside_a_jump(dim, N, count, jump):
    """Patches with an oblique jump of density and pressure, errors by subcell."""
    import torch
    rng = np.random.default_rng(3 * N + dim)
    L, Ns, nv = 2 * N + 7, 2 * N + 1, dim + 2
    shape = (count,) + (L,) * dim
    one = (count,) + (1,) * dim
    x = sum(rng.normal(size=one) * (np.arange(L) - L / 2 + 0.5).reshape((1,) * (1 + k) + (L,) + (1,) * (dim - 1 - k))
            for k in range(dim))
    side = x < rng.uniform(-1, 1, one)
    rho = np.where(side, 1.0, 1.0 / jump) * rng.uniform(0.98, 1.02, shape)
    p = np.where(side, 1.0, 1.0 / jump) * rng.uniform(0.98, 1.02, shape)
    P = euler.prim_to_cons(rho, [rng.uniform(-0.2, 0.2, shape) for _ in range(dim)], p, GAMMA)
    h = [0.01 * (1 + 0.3 * k) for k in range(dim)]
    dt = 0.1 * h[0] / dim
    ref, _ = ader_weno(P, dt, h, GAMMA, dim)
    q = np.transpose(P, [1, 0] + list(range(dim + 1, 1, -1))).reshape(count, nv, -1)
    q = torch.from_numpy(np.ascontiguousarray(q)).cuda()
    v = torch.empty((count, nv, Ns ** dim), dtype=torch.float64, device="cuda")
    rc, msg = adg.subcell_update_noalloc(dim, N, GAMMA, h, dt, q.data_ptr(), count, v.data_ptr())
    assert rc == adg.OK, msg
    torch.cuda.synchronize()
    got = np.transpose(v.cpu().numpy().reshape((count, nv) + (Ns,) * dim), [1, 0] + list(range(dim + 1, 1, -1)))
    scale = _nearby(P, range(2, 2 + dim))[(slice(None),) * 2 + (slice(3, 3 + Ns),) * dim]
    scale[1:1 + dim] = scale[1:1 + dim].max(axis=0)
    ok = np.isfinite(ref)
    assert ok.mean() > 0.9 and np.array_equal(ok, np.isfinite(got))
    err = np.abs(got - ref)[ok] / scale[ok]
    assert err.max() <= RTOL, err.max()


@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("N,n", [(1, 16), (2, 14), (5, 12), (7, 10)])
def test_step_over_six_decades(N, n, force):
    """A smooth periodic flow whose density and pressure span six decades, errors by cell."""
    g = Grid((n, 4), (0.0, 0.0), (1.0 / n, 0.25), (0, 0, 0, 0))
    sch = Scheme(g, N, GAMMA)
    xi = sch.basis.xi
    x = (np.arange(n).reshape(n, 1, 1, 1) + xi.reshape(1, 1, -1, 1)) / n
    y = 0.25 * (np.arange(4).reshape(1, 4, 1, 1) + xi.reshape(1, 1, 1, -1))
    f = np.exp(-0.5 * np.log(1e6) * (1 - np.cos(2 * np.pi * x)) / 2 * 2) * (1 + 0.1 * np.sin(2 * np.pi * y))
    one = np.ones_like(f)
    U = euler.prim_to_cons(f, [0.3 * one, -0.2 * one], f, GAMMA)
    st = State(U, np.zeros((n, 4), dtype=np.int32), np.full((4, n, 4) + (sch.Ns,) * 2, np.nan))
    dt = 0.3 * stable_dt(sch, st, 1.0 / (2 * (2 * N + 1)))
    ref, _ = step(sch, st, dt, force_all=force)
    s = adg.Solver(2, (n, 4), (0.0, 0.0), (1.0 / n, 0.25), (0, 0, 0, 0), N, GAMMA, adg.PREC_FP64)
    s.set_option(adg.OPT_FORCE_LIMITER, int(force))
    load_state(s, sch, st)
    s.step(dt)
    d, b, _ = s.read_full()
    assert s.status() == adg.OK
    s.close()
    got, beta = from_abi(d, 2, (n, 4), N + 1), beta_from_abi(b, (n, 4))
    assert np.array_equal(beta, ref.beta)
    cell = np.abs(U).max(axis=(3, 4))
    cell[1:3] = cell[1:3].max(axis=0)
    scale = _nearby(cell, (1, 2))
    err = np.abs(got - ref.U).max(axis=(3, 4)) / scale
    assert err.max() <= RTOL, err.max()
