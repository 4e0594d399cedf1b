"""GPU: the standalone operators where their launch rules branch.  The
sensitivity image by ring-pair profiles (rings that are copies of each other,
z-principal ring pairs, a displaced ring, non-TOF, planes in several groups)
against the FP64 oracle; projections of many events (TOF weights from a table
per block; from 16 384 events on 3D grids by the table projector's walk)
against the same events in small calls (the event kernel, an erf per sample)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2201_05497_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lm():
    from paper_2201_05497_gb300 import build, lm as _lm
    build.build()
    _lm.load_library()
    return _lm


# (rings, crystals, radius, pitch), grid, voxel size, TOF bins, displaced crystal
SENS = {
    "cylinder": ((9, 40, 100.0, 7.0), (24, 21, 16), 6.0, 15, False),
    "non_tof": ((9, 40, 100.0, 7.0), (24, 21, 16), 6.0, 0, False),
    "z_principal": ((20, 24, 40.0, 8.0), (16, 18, 30), 4.0, 9, False),
    "displaced": ((6, 32, 100.0, 7.0), (20, 20, 9), 7.0, 9, True),
    "plane_groups": ((20, 16, 150.0, 9.0), (270, 9, 20), 1.0, 9, False),
}


@pytest.mark.parametrize("name", sorted(SENS))
def test_sens_matches_oracle(lm, name):
    (rings, xtal, radius, pitch), n, h, bins, displaced = SENS[name]
    sc = S.Scanner(rings, xtal, radius, pitch)
    g = S.Grid(n, (h, h, h))
    tof = (20.0, 18.0, 3.0, bins)
    tab = sc.crystal_table().copy()
    if displaced:
        tab[2 * xtal + 5] += np.float32([1.5, -0.7, 0.4])
    lf = np.random.default_rng(3).uniform(0.2, 1.0, sc.n_lor).astype(np.float32)
    geo_o = O.Geometry(tab, rings, xtal, g.n, g.h, g.origin, tof)
    geo_g = lm.Geometry(torch.from_numpy(tab).cuda(), rings, xtal, g.n, g.h, g.origin, *tof)
    s_or = O.sens(geo_o, lf)
    for ws in (True, False):
        s = lm.sens(geo_g, torch.from_numpy(lf).cuda(), use_workspace=ws).cpu().numpy()
        assert np.linalg.norm(s - s_or) <= 1e-5 * np.linalg.norm(s_or), ws


# scanner (rings, crystals, radius, pitch), grid, voxel size, TOF bins
PROJ = {
    "2d": ((1, 128, 150.0, 1.0), (41, 37, 1), 5.0, 27),
    "rows": ((8, 96, 150.0, 8.0), (41, 37, 14), 5.0, 27),
    "bricks": ((8, 96, 150.0, 8.0), (44, 36, 14), 5.0, 27),
    "non_tof": ((8, 96, 150.0, 8.0), (44, 36, 14), 5.0, 0),
    "non_tof_many_planes": ((8, 96, 150.0, 8.0), (180, 36, 14), 1.0, 0),
    "z_principal": ((60, 48, 60.0, 6.0), (24, 20, 80), 4.0, 27),
}


@pytest.mark.parametrize("name", sorted(PROJ))
def test_many_events_equal_few(lm, name):
    """The table interpolates the TOF kernel to 1e-7 of its peak and erf
    carries as much, so a projection moves by at most 4e-7 of the largest
    per tap."""
    (rings, xtal, radius, pitch), n_g, h, bins = PROJ[name]
    sc = S.Scanner(rings, xtal, radius, pitch)
    g = S.Grid(n_g, (h, h, h))
    tof = S.tof_400ps(bins, 600.0 / 27)
    n = 90000
    ev = S.uniform_events(sc, tof, n, 5)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    dev = lm.DeviceEvents.from_numpy(ev)
    rng = np.random.default_rng(2)
    x = torch.from_numpy(rng.uniform(0.1, 1, geo.V).astype(np.float32)).cuda()
    v = torch.from_numpy(rng.normal(size=n).astype(np.float32)).cuda()
    p = lm.fwd(geo, x, dev).double()
    b = lm.back(geo, v, dev).double()
    ps, bs = [], torch.zeros(geo.V, dtype=torch.float64, device="cuda")
    for s in range(0, n, 6000):
        part = lm.DeviceEvents(*[t[s:s + 6000].contiguous() for t in (dev.det1, dev.det2, dev.tof, dev.corr, dev.contam)])
        ps.append(lm.fwd(geo, x, part).double())
        bs += lm.back(geo, v[s:s + 6000].contiguous(), part).double()
    ps = torch.cat(ps)
    assert float((p - ps).abs().max()) <= 4e-7 * float(ps.abs().max()) * 4  # four taps
    assert float((b - bs).norm() / bs.norm()) <= 2e-6


def test_non_finite_stays_with_its_weight(lm):
    """A voxel of weight 0 does not enter a projection, nor does an event's
    value enter a voxel of weight 0, whatever they hold: an infinite voxel
    or value touches the same elements as with few events."""
    sc = S.Scanner(9, 64, 150.0, 5.0)
    g = S.Grid((44, 36, 9), (5.0, 5.0, 5.0))  # rings on slice centres: the upper neighbour's weight is often 0
    tof = S.tof_400ps(27, 600.0 / 27)
    n = 20000
    ev = S.uniform_events(sc, tof, n, 8)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    dev = lm.DeviceEvents.from_numpy(ev)
    x = torch.ones(geo.V, device="cuda")
    x[44 * 36 * 4:44 * 36 * 5] = float("inf")
    v = torch.ones(n, device="cuda")
    v[::1000] = float("inf")
    p = torch.isfinite(lm.fwd(geo, x, dev))
    b = lm.back(geo, v, dev)
    ps, bs = [], torch.zeros(geo.V, device="cuda")
    for s in range(0, n, 5000):
        part = lm.DeviceEvents(*[t[s:s + 5000].contiguous() for t in (dev.det1, dev.det2, dev.tof, dev.corr, dev.contam)])
        ps.append(torch.isfinite(lm.fwd(geo, x, part)))
        bs = lm.back(geo, v[s:s + 5000].contiguous(), part, img=bs)
    assert bool((p == torch.cat(ps)).all()) and not bool(p.all()) and bool(p.any())
    assert not bool(torch.isnan(b).any()) and bool((torch.isinf(b) == torch.isinf(bs)).all())
