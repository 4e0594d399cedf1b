"""GPU: the table projector's walk (two lanes per plane over z-pair images)
against the direct event kernel on the grids where its branches differ:
bricked and row layouts, events with more planes than a warp keeps in
registers, z-principal events, one-slice-deep and very small grids.  Same
samples and weights, sums in another order: 1e-5 relative L2 as for the other
comparisons of the two projectors."""
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


# (rings, crystals, radius, pitch), grid, voxel size, events
CASES = {
    "bricks": ((12, 96, 150.0, 6.0), (48, 44, 20), 4.0, 20000),
    "rows": ((12, 96, 150.0, 6.0), (45, 38, 21), 4.0, 20000),
    "bricks_plain_passes": ((12, 96, 150.0, 6.0), (32, 28, 16), 5.0, 20000),
    "many_planes": ((8, 96, 150.0, 6.0), (132, 120, 16), 1.0, 8000),
    "z_principal": ((60, 48, 60.0, 6.0), (40, 36, 90), 2.5, 20000),
    "z_principal_rows": ((60, 48, 60.0, 6.0), (39, 35, 90), 2.5, 20000),
    "two_slices": ((4, 96, 150.0, 3.0), (44, 40, 2), 4.0, 3000),
    "few_events": ((12, 96, 150.0, 6.0), (48, 44, 20), 4.0, 37),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_table_walk_matches_direct(lm, name):
    (rings, xtal, radius, pitch), n, h, n_ev = CASES[name]
    sc = S.Scanner(rings, xtal, radius, pitch)
    g = S.Grid(n, (h, h, h))
    tof = S.tof_400ps(27, 600.0 / 27)
    ev = S.uniform_events(sc, tof, n_ev, 4)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), rings, xtal, g.n, g.h, g.origin, tof.sigma, tof.bin,
                      tof.n_sigma, tof.n_bins)
    pe = lm.event_setup(geo, lm.DeviceEvents.from_numpy(ev), 3)
    sens = lm.sens(geo)
    rng = np.random.default_rng(7)
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda() * (n_ev / float(sens.sum()))
    out = {}
    for proj in ("direct", "table"):
        st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.03, n_subsets=3, knorm=H.knorm_closed(n), projector=proj, group=32)
        assert st.tuning()["projector"] == proj
        st.updates([0, 3, 1])
        st.updates([3, 2, 0])
        out[proj] = (st.x().cpu().numpy(), st.y().cpu().numpy(), st.z().cpu().numpy(), st.objective())
        st.close()
    for k in range(3):
        assert H.rel_l2(out["table"][k], out["direct"][k]) < 1e-5, k
    assert abs(out["table"][3] - out["direct"][3]) <= 1e-5 * abs(out["direct"][3])
