"""GPU: the FP64 reconstruction where one stencil is flat and another crosses a jump whose
oscillation indicator lies near the end of the FP64 range, or beyond it: the flat one takes all of
the weight."""
import numpy as np
import pytest

from paper_1406_7416_gb300 import adg, build_lib

pytestmark = pytest.mark.gpu
GAMMA = 1.4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    adg.load_library()


@pytest.mark.parametrize("jump", [1e8, 1e140, 1e147, 1e148, 1e153, 1e160])
@pytest.mark.parametrize("dim,N", [(2, 1), (2, 3), (3, 1)])
def test_flat_stencils_take_the_weight(dim, N, jump):
    """A gas at rest with a jump of the energy and a step too short to change anything: the update
    returns the averages.  A reconstruction from across the jump would have a negative pressure
    beside it, and no number for its sound speed."""
    import torch
    L, Ns, nv = 2 * N + 7, 2 * N + 1, dim + 2
    P = np.zeros((L - 5, nv) + (L,) * dim)
    P[:, 0] = 1.0
    for c in range(L - 5):                          # the jump between x = c + 2 and c + 3
        P[c, dim + 1] = np.where(np.arange(L) < c + 3, 2.5, 2.5 * jump)
    q = torch.from_numpy(P.reshape(L - 5, nv, -1).copy()).cuda()
    v = torch.empty((L - 5, nv, Ns ** dim), dtype=torch.float64, device="cuda")
    dt = 0.01 / jump ** 1.5 / 1e20
    rc, msg = adg.subcell_update_noalloc(dim, N, GAMMA, [0.01] * dim, dt, q.data_ptr(), L - 5, v.data_ptr())
    assert rc == adg.OK, msg
    torch.cuda.synchronize()
    want = P[(slice(None),) * 2 + (slice(3, 3 + Ns),) * dim].reshape(L - 5, nv, -1)
    got = v.cpu().numpy()
    assert np.isfinite(got).all()
    # beside a step of 1e-20 of the limit, the rounding of one difference
    np.testing.assert_allclose(got[:, [0, dim + 1]], want[:, [0, dim + 1]], rtol=1e-15)
