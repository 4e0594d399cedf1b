"""GPU: device arrays of the caller that start at any float.  A directional-TV
field at an odd offset gives the aligned field's iterates bit for bit
(deterministic mode), in the TMA-staged prior pass and in the event kernel's
prior branch; EM-TV iterates into an image at an odd offset equal the aligned
image's to rounding (12 iterations of about ten roundings each, no atomics)."""
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


def small_frame(lm, n=(44, 40, 12), n_ev=4000):
    sc = S.Scanner(6, 96, 150.0, 6.0)
    g = S.Grid(n, (4.0, 4.0, 4.0))
    tof = S.tof_400ps(27, 600.0 / 27)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    ev = lm.DeviceEvents.from_numpy(S.uniform_events(sc, tof, n_ev, 4))
    return geo, ev


def shifted(t, offset):
    """A contiguous copy of t that starts `offset` elements after a 256-byte boundary."""
    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    view = buf[offset:offset + t.numel()]
    view.copy_(t)
    assert (view.data_ptr() & 15) == 4 * offset % 16
    return view


@pytest.mark.parametrize("image_kernel,kind", [(1, "plain"), (2, "tma"), (3, "tma_data")])
def test_directional_field_at_any_float(lm, image_kernel, kind):
    geo, ev = small_frame(lm)
    pe = lm.event_setup(geo, ev, 3)
    sens = lm.sens(geo)
    rng = np.random.default_rng(7)
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda() * (ev.n / float(sens.sum()))
    xi = lm.dtv_field(geo, torch.from_numpy(rng.uniform(0, 1, geo.V).astype(np.float32)).cuda(), 0.05)
    out = []
    for offset in range(4):
        st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.1, n_subsets=3, knorm=H.knorm_closed(geo.n), deterministic=True,
                        image_kernel=image_kernel, group=32, xi=shifted(xi, offset))
        assert st.tuning()["image_kernel"] == kind
        st.epoch([3, 0, 3, 3, 1, 2])
        out.append([t.cpu().numpy() for t in (st.x(), st.z(), st.w())])
        st.close()
    assert np.abs(out[0][2]).max() > 0
    for offset in (1, 2, 3):
        for a, b in zip(out[offset], out[0]):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [(44, 40, 12), (42, 40, 12)])
def test_denoised_image_at_any_float(lm, n):
    geo, _ = small_frame(lm, n)
    rng = np.random.default_rng(8)
    z = torch.from_numpy(rng.uniform(0, 2, geo.V).astype(np.float32)).cuda()
    w = torch.from_numpy(rng.uniform(0.5, 3, geo.V).astype(np.float32)).cuda()
    want = lm.emtv_denoise(geo, z, w, 12, H.knorm_closed(n)).cpu().numpy()
    for offset in (1, 2, 3):
        u = lm.emtv_denoise(geo, z, w, 12, H.knorm_closed(n), out=shifted(z, offset))
        assert H.rel_l2(u.cpu().numpy(), want) < 1e-5
