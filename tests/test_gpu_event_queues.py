"""GPU: the event kernel's two work counters.  Launches of up to eight chunks per
warp (data updates: 64 events; 16 and 32 lanes per event) draw them from a counter
per block, larger ones and 8 lanes from the launch's; both sides of the line give the same
sums to rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_05497_gb300 import synth as S
from tests import _helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lm():
    from paper_2201_05497_gb300 import build, lm as _lm
    build.build()
    _lm.load_library()
    return _lm


def frame(lm, two_d, n_ev):
    sc = S.Scanner(1, 128, 150.0, 1.0) if two_d else S.Scanner(8, 96, 150.0, 8.0)
    g = S.Grid((44, 40, 1) if two_d else (44, 36, 14), (5.0, 5.0, 5.0))
    tof = S.tof_400ps(27, 600.0 / 27)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    return geo, lm.DeviceEvents.from_numpy(S.uniform_events(sc, tof, n_ev, 5))


@pytest.mark.parametrize("two_d", [False, True])
@pytest.mark.parametrize("n_ev", [1, 37, 60000, 300000])
def test_data_updates_agree_over_widths(lm, two_d, n_ev):
    geo, ev = frame(lm, two_d, n_ev)
    pe = lm.event_setup(geo, ev, 1)
    sens = lm.sens(geo) + 1.0
    rng = np.random.default_rng(3)
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda() * (ev.n / float(sens.sum()))
    out = []
    for group in (8, 16, 32):
        st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.03, n_subsets=1, knorm=H.knorm_closed(geo.n), projector="direct",
                        group=group)
        st.updates([0, 1, 0])
        out.append([t.cpu().numpy() for t in (st.x(), st.y(), st.z())])
        st.close()
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert H.rel_l2(a, b) < 1e-5


@pytest.mark.parametrize("two_d", [False, True])
def test_em_step_equals_its_parts(lm, two_d):
    """The EM back-projection is a sum over events: of 1 000 000 in one launch, of
    200 000 in each of five."""
    geo, ev = frame(lm, two_d, 1000000)
    rng = np.random.default_rng(4)
    sens = torch.from_numpy(rng.uniform(1, 2, geo.V).astype(np.float32)).cuda()
    x = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda()
    whole = lm.emtv_em_step(geo, ev, 1, sens, x).double()
    parts = torch.zeros_like(whole)
    for s in range(0, ev.n, 200000):
        part = lm.DeviceEvents(*[t[s:s + 200000].contiguous() for t in (ev.det1, ev.det2, ev.tof, ev.corr, ev.contam)])
        parts += lm.emtv_em_step(geo, part, 1, sens, x).double()
    assert float((whole - parts).norm() / parts.norm()) < 2e-6
