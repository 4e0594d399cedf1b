"""GPU: the sensitivity image where its rule for ring-pair profiles branches.
A scanner longer than wide (most LORs go one by one, by warps that hold no
planes), a grid too fine axially for the profiles (LOR by LOR throughout), against
the FP64 oracle; and factors that are not finite, which stay with the voxels
that their LORs touch."""
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


def geometry(lm, scanner, n, h, bins):
    sc = S.Scanner(*scanner)
    g = S.Grid(n, (h, h, h))
    tab = sc.crystal_table()
    args = (sc.n_rings, sc.n_xtal, g.n, g.h, g.origin)
    return sc, O.Geometry(tab, *args, (20.0, 18.0, 3.0, bins)), lm.Geometry(torch.from_numpy(tab).cuda(), *args, 20.0, 18.0,
                                                                            3.0, bins)


# (rings, crystals, radius, pitch), grid, voxel size, TOF bins
CASES = {
    "long": ((72, 24, 40.0, 3.1), (16, 18, 100), 2.0, 9),
    "long_non_tof": ((60, 24, 40.0, 3.1), (33, 18, 90), 2.0, 0),
    "fine_axial": ((18, 32, 100.0, 3.1), (96, 90, 600), 1.0, 9),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_sens_matches_oracle(lm, name):
    sc, geo_o, geo = geometry(lm, *CASES[name])
    lf = np.random.default_rng(3).uniform(0.2, 1.0, sc.n_lor).astype(np.float32)
    want = O.sens(geo_o, lf)
    got = lm.sens(geo, torch.from_numpy(lf).cuda()).cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_factor_stays_with_its_lor(lm, value):
    """Rings on slice centres, so that upper neighbours weigh 0; one factor
    that is not finite within a ring, one between two rings."""
    sc, _, geo = geometry(lm, (9, 40, 100.0, 5.0), (24, 21, 9), 5.0, 15)
    lf = torch.ones(sc.n_lor, device="cuda")
    bad = torch.zeros(sc.n_lor, device="cuda")
    for q, r1, r2 in ((18 * 40 + 7, 4, 4), (15 * 40 + 33, 1, 6)):  # nearly opposite crystals
        bad[q * 81 + r1 * 9 + r2] = 1.0
    touched = lm.sens(geo, bad) > 0
    lf[bad > 0] = value
    s = lm.sens(geo, lf)
    assert bool(touched.any()) and bool((torch.isfinite(s) == ~touched).all())
