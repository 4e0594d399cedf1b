"""GPU: non-finite values in the table projector's data updates.  A voxel of
weight 0 does not enter an event's projection and an event's value does not
enter a voxel of weight 0, whatever they hold.  Rings on slice centres and events
within one ring: each event lies in one slice, its upper neighbour weighs 0."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_05497_gb300 import synth as S
from tests import _helpers as H

pytestmark = pytest.mark.gpu

BAD = 4  # the slice that holds infinities


@pytest.fixture(scope="module")
def lm():
    from paper_2201_05497_gb300 import build, lm as _lm
    build.build()
    _lm.load_library()
    return _lm


@pytest.mark.parametrize("n,h", [((44, 40, 9), 5.0), ((43, 39, 9), 5.0), ((180, 160, 9), 1.25)])
def test_infinite_slice_stays_its_own(lm, n, h):
    sc = S.Scanner(9, 64, 150.0, 5.0)
    tof = S.tof_400ps(27, 600.0 / 27)
    ev = S.uniform_events(sc, tof, 6000, 8)
    ring = np.arange(ev.n) % 9
    ev.det1, ev.det2 = (ring * 64 + ev.det1 % 64).astype(np.int32), (ring * 64 + ev.det2 % 64).astype(np.int32)
    g = S.Grid(n, (h, h, 5.0))
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    dev = lm.DeviceEvents.from_numpy(ev)
    inside = lm.fwd(geo, torch.ones(geo.V, device="cuda"), dev) > 0
    pe = lm.event_setup(geo, dev, 1)  # one subset: the events keep their order
    sens = lm.sens(geo)
    x0 = torch.full((geo.V,), ev.n / float(sens.sum()), device="cuda")
    st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.03, n_subsets=1, gamma=1.0, knorm=H.knorm_closed(n), projector="table",
                    group=32)
    x1 = x0.view(n[2], -1).clone()
    x1[BAD] = float("inf")
    st.reinit(x1.view(-1))
    st.updates([0])
    y, z = st.y(), st.z().view(n[2], -1)
    st.close()
    mine = torch.from_numpy(ring == BAD).cuda() & inside
    assert bool(mine.any()) and not bool(torch.isfinite(y[mine]).any())  # infinite projection, undefined dual
    assert bool(torch.isfinite(y[~mine]).all())
    assert not bool(torch.isfinite(z[BAD]).all())
    assert bool(torch.isfinite(torch.cat([z[:BAD], z[BAD + 1:]])).all())


def test_batch_frame_with_an_infinite_slice(lm):
    """The batch's kernel: a frame with infinities beside one without."""
    n, h = (44, 40, 9), 5.0
    sc = S.Scanner(9, 64, 150.0, 5.0)
    tof = S.tof_400ps(27, 600.0 / 27)
    ev = S.uniform_events(sc, tof, 6000, 8)
    ring = np.arange(ev.n) % 9
    ev.det1, ev.det2 = (ring * 64 + ev.det1 % 64).astype(np.int32), (ring * 64 + ev.det2 % 64).astype(np.int32)
    g = S.Grid(n, (h, h, 5.0))
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    sens = lm.sens(geo)
    x0 = torch.full((geo.V,), ev.n / float(sens.sum()), device="cuda")
    x1 = x0.view(n[2], -1).clone()
    x1[BAD] = float("inf")
    batch, frames = lm.Batch(2, 1), []
    for i, x in enumerate((x1.view(-1), x0)):
        pe = lm.event_setup(geo, lm.DeviceEvents.from_numpy(ev), 1)
        frames.append(lm.LMSPDHG(geo, pe, sens, x, beta=0.03, n_subsets=1, gamma=1.0, knorm=H.knorm_closed(n),
                                 projector="table", group=32))
        batch.set(i, frames[-1])
    batch.epoch(np.array([[0, 1], [0, 1]], np.uint16))
    y, z = frames[0].y(), frames[0].z().view(n[2], -1)
    other = torch.from_numpy(ring != BAD).cuda()
    assert bool(torch.isfinite(y[other]).all()) and not bool(torch.isfinite(y[~other]).all())
    assert bool(torch.isfinite(frames[1].y()).all()) and bool(torch.isfinite(frames[1].z()).all())
    far = [s for s in range(9) if abs(s - BAD) > 1]  # (the prior update reaches one slice further)
    assert bool(torch.isfinite(z[far]).all())
