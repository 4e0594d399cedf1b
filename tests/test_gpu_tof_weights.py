"""GPU: TOF weights of the standalone projections against the erf difference in
64 bits, for narrow and wide cuts and for few and many events of a call.

Every number of the geometry is exact in float32 (lines along x of length 512
mm through voxel centres, centres at multiples of 1/64 mm, bins of 22 mm), so
a projection of one voxel is the sample length times the weight, and what
is left is: two erff of 2 ulp each (their documented bound, values up to 1) and
three roundings of an argument z, where |z erf'(z)| <= 0.484.  With the factor
1/2 of the weight that is 2 * 2^-24 + 0.484 * 3 * 2^-24 = 3.5 * 2^-24 at most,
plus the roundings of the products (4 * 2^-24 of a weight below 1/3).  The walk's
expansion about the nodes of a table has the same two roundings of its nodes and a
remainder below 2^-26."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = (3.5 + 1.4) * 2.0 ** -24
SIGMA, BIN, NB, H = float(np.float32(25.46)), 22.0, 41, 2.0
N = (64, 32, 16)


@pytest.fixture(scope="module")
def lm():
    from paper_2201_05497_gb300 import build, lm as _lm
    build.build()
    _lm.load_library()
    return _lm


def setup(lm, n_sigma, copies):
    rows = N[1] * N[2]
    j = np.arange(rows)
    d = j / 64.0
    y, z = H * (j % N[1]) - 32.0, H * (j // N[1]) - 16.0
    tab = np.concatenate([np.stack([-256.0 + d, y, z], 1), np.stack([256.0 + d, y, z], 1)]).astype(np.float32)
    geo = lm.Geometry(torch.from_numpy(tab).cuda(), 16, 2 * rows // 16, N, (H, H, H), (-64.0, -32.0, -16.0), SIGMA, BIN,
                      n_sigma, NB)
    row = np.tile(np.repeat(j, NB), copies)
    m = np.tile(np.tile(np.arange(NB) - NB // 2, rows), copies)
    t = lambda a, dt: torch.from_numpy(a.astype(dt)).cuda()  # noqa: E731
    ev = lm.DeviceEvents(t(row, np.int32), t(row + rows, np.int32), t(m, np.int16), None, None)
    return geo, ev, row, m


def weight(tau, n_sigma):
    """The weight in 64 bits, and where |tau| is too near the cut to decide."""
    s = math.sqrt(2.0) * SIGMA
    erf = np.vectorize(math.erf)
    w = 0.5 * (erf((tau + BIN / 2) / s) - erf((tau - BIN / 2) / s))
    return np.where(np.abs(tau) <= n_sigma * SIGMA, w, 0.0), np.abs(np.abs(tau) - n_sigma * SIGMA) < 1e-3


@pytest.mark.parametrize("n_sigma", [3.0, 5.0, 10.0, 12.0])
@pytest.mark.parametrize("workspace", [True, False])  # the walk over z pairs / the event kernel
def test_weights_of_many_events(lm, n_sigma, workspace):
    geo, ev, row, m = setup(lm, n_sigma, 3)
    assert ev.n > 60000
    for plane in (5, 33):
        x = torch.zeros(N[2], N[1], N[0], device="cuda")
        x[:, :, plane] = 1.0
        p = lm.fwd(geo, x.reshape(-1), ev, use_workspace=workspace).double().cpu().numpy()
        want, edge = weight(-64.0 + H * plane - row / 64.0 - m * BIN, n_sigma)
        assert np.abs(p / H - want)[~edge].max() <= TOL
    # one event with a value per row: each voxel receives one weight
    pick = np.arange(ev.n) < N[1] * N[2] * NB
    pick &= m == row % NB - NB // 2
    img = lm.back(geo, torch.from_numpy(pick.astype(np.float32)).cuda(), ev, use_workspace=workspace)
    img = img.double().cpu().numpy().reshape(N[1] * N[2], N[0])
    j = np.arange(N[1] * N[2])[:, None]
    want, edge = weight(-64.0 + H * np.arange(N[0])[None] - j / 64.0 - (j % NB - NB // 2) * BIN, n_sigma)
    assert np.abs(img / H - want)[~edge].max() <= TOL and want.max() > 0.3
