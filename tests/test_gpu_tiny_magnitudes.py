"""GPU: the FP64 subcell update at magnitudes whose fluxes lie below the range that the fixed-point
products work in.  The Euler fluxes are homogeneous of degree one and the variations here are far
below the reconstruction's 1e-14, so the update scales with a power of two: from 2^-60, 2^-970 and
2^-1000 the same patch gives the same result.  (Velocities of 1e-8 keep the squares of momenta,
which underflow at the lower scales, below the last place of the pressure.)"""
import numpy as np
import pytest

from paper_1406_7416_gb300 import adg, build_lib

pytestmark = pytest.mark.gpu
GAMMA = 1.4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


def _update(P, dim, N):
    import torch
    count, nv, Ns = P.shape[0], dim + 2, 2 * N + 1
    h = [0.01 * (1 + 0.3 * k) for k in range(dim)]
    q = torch.from_numpy(np.ascontiguousarray(P)).cuda()
    v = torch.empty((count, nv, Ns ** dim), dtype=torch.float64, device="cuda")
    rc, msg = adg.subcell_update_noalloc(dim, N, GAMMA, h, 0.1 * h[0] / dim, q.data_ptr(), count, v.data_ptr())
    assert rc == adg.OK, msg
    torch.cuda.synchronize()
    return v.cpu().numpy()


@pytest.mark.parametrize("exp", [-900, -970, -1000])
@pytest.mark.parametrize("dim,N", [(2, 1), (2, 4), (3, 1), (3, 2)])
def test_update_scales(dim, N, exp):
    rng = np.random.default_rng(dim + N)
    count, L = 3, 2 * N + 7
    P = np.ones((count, dim + 2, L ** dim))
    P[:, dim + 1] = 1.0 / (GAMMA - 1.0)
    P *= 1.0 + 1e-8 * rng.uniform(-1, 1, P.shape)
    P[:, 1:dim + 1] = 1e-8 * rng.uniform(-1, 1, P[:, 1:dim + 1].shape)
    P[1, 2] = 0.0                                   # and a momentum at rest
    # 44 bits of each value from 2^0 down: the same patch at every scale
    P = np.round(np.ldexp(P, 44))
    a = np.ldexp(_update(np.ldexp(P, -44 - 60), dim, N), 60)
    b = np.ldexp(_update(np.ldexp(P, -44 + exp), dim, N), -exp)
    assert np.isfinite(a).all()
    inner = (slice(3, 3 + 2 * N + 1),) * dim
    before = np.ldexp(P, -44).reshape((count, dim + 2) + (L,) * dim)[(slice(None),) * 2 + inner]
    assert np.abs(a - before.reshape(a.shape)).max() > 1e-10
    # each step of the update rounds at 1e-16 of values up to 2.5, or in subnormal values at
    # 2^-1074 (2^-74 of the scale at the lowest): fewer than 1e3 of them
    err = np.abs(b - a).max()
    assert err <= 1e-12, err
