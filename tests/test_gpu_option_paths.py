"""GPU: options together with the paths they now take.  The table projector's
pair images under the directional TV and every image pass against the direct
kernel; the operators with workspaces that do not hold a pair image; the
one-voxel passes of small 2D images against the tiled ones without atomics in
between, bit for bit."""
import ctypes as C

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


def frame(lm, n, n_ev, seed=4):
    sc = S.Scanner(12, 96, 150.0, 6.0) if n[2] > 1 else S.Scanner(1, 96, 150.0, 1.0)
    g = S.Grid(n, (4.0, 4.0, 4.0))
    tof = S.tof_400ps(27, 600.0 / 27)
    geo = lm.Geometry(torch.from_numpy(sc.crystal_table()).cuda(), sc.n_rings, sc.n_xtal, g.n, g.h, g.origin, tof.sigma,
                      tof.bin, tof.n_sigma, tof.n_bins)
    return geo, lm.DeviceEvents.from_numpy(S.uniform_events(sc, tof, n_ev, seed))


@pytest.mark.parametrize("n,image_kernel,kind", [((48, 44, 20), 0, "tma"), ((48, 44, 20), 3, "tma_data"),
                                                 ((48, 44, 20), 1, "plain"), ((45, 38, 21), 0, "plain")])
@pytest.mark.parametrize("dtv", [False, True])
def test_table_under_options_matches_direct(lm, n, image_kernel, kind, dtv):
    geo, ev = frame(lm, n, 20000)
    pe = lm.event_setup(geo, ev, 3)
    sens = lm.sens(geo)
    rng = np.random.default_rng(7)
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda() * (ev.n / float(sens.sum()))
    xi = lm.dtv_field(geo, torch.from_numpy(rng.uniform(0, 1, geo.V).astype(np.float32)).cuda(), 0.05) if dtv else None
    out = {}
    for proj in ("direct", "table"):
        st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.03, n_subsets=3, knorm=H.knorm_closed(n), projector=proj, group=32, xi=xi,
                        image_kernel=image_kernel)
        t = st.tuning()
        assert (t["projector"], t["image_kernel"]) == (proj, kind)
        st.epoch([0, 3, 1, 3, 2, 0])
        st.updates([3, 2, 3])
        out[proj] = [v.cpu().numpy() for v in (st.x(), st.y(), st.z(), st.w())] + [st.objective()]
        st.close()
    for k in range(3):
        assert H.rel_l2(out["table"][k], out["direct"][k]) < 1e-5, k
    assert H.rel_l2(out["table"][3], out["direct"][3]) < H.REL_L2_IMAGE  # differences of neighbouring x
    assert abs(out["table"][4] - out["direct"][4]) <= 1e-5 * abs(out["direct"][4])


@pytest.mark.parametrize("n", [(44, 36, 14), (41, 37, 14)])
def test_operator_workspaces(lm, n):
    """No workspace, one copy's (4 bytes per voxel), a pair image's at an odd
    float and at 16 bytes: the same projections from the event kernel and the walk."""
    geo, ev = frame(lm, n, 20000)
    L, V, d = lm.load_library(), geo.V, ev.desc()
    rng = np.random.default_rng(2)
    x = torch.from_numpy(rng.uniform(0.1, 1, V).astype(np.float32)).cuda()
    v = torch.from_numpy(rng.normal(size=ev.n).astype(np.float32)).cuda()
    need = int(L.lm_fwd_workspace_bytes(C.byref(geo.g)))
    assert need == int(L.lm_back_workspace_bytes(C.byref(geo.g), 0)) >= 8 * V
    one = (4 * V + 255) // 256 * 256
    buf = torch.empty(need + 512, dtype=torch.uint8, device="cuda")
    guard = 0xA5
    got = []
    for offset, size in ((0, 0), (0, one), (4, one), (4, need), (16, need), (0, need)):
        buf.fill_(guard)
        p, b = torch.empty(ev.n, device="cuda"), torch.zeros(V, device="cuda")
        ws = C.c_void_p(buf.data_ptr() + offset) if size else None
        lm._check(L.lm_fwd(C.byref(geo.sc), C.byref(geo.g), C.byref(geo.tof), x.data_ptr(), C.byref(d), p.data_ptr(), ws,
                           size, lm._stream()))
        lm._check(L.lm_back(C.byref(geo.sc), C.byref(geo.g), C.byref(geo.tof), C.byref(d), v.data_ptr(), b.data_ptr(), 0, ws,
                            size, lm._stream()))
        # nothing outside the workspace is written
        assert bool((buf[:offset] == guard).all()) and bool((buf[offset + size:] == guard).all()), (offset, size)
        got.append((p.cpu().numpy(), b.cpu().numpy()))
    for p, b in got[1:]:
        assert H.rel_l2(p, got[0][0]) < 2e-6 and H.rel_l2(b, got[0][1]) < 2e-6


@pytest.mark.parametrize("n_ev", [20000, 24576, 30000])
def test_forward_on_both_sides_of_the_voxel_line(lm, n_ev):
    """6.3e6 voxels: 24 576 events are one per 256 voxels, from where the walk
    over z pairs serves a forward projection; against small calls."""
    geo, ev = frame(lm, (256, 256, 96), n_ev)
    x = torch.from_numpy(np.random.default_rng(2).uniform(0.1, 1, geo.V).astype(np.float32)).cuda()
    p = lm.fwd(geo, x, ev)
    for s in range(0, n_ev, 6000):
        part = lm.DeviceEvents(*[t[s:s + 6000].contiguous() for t in (ev.det1, ev.det2, ev.tof, ev.corr, ev.contam)])
        q = lm.fwd(geo, x, part)
        assert float((p[s:s + 6000] - q).abs().max()) <= 2e-6 * float(p.abs().max())


@pytest.mark.parametrize("n", [(2, 3, 1), (33, 31, 1), (64, 48, 1), (362, 362, 1)])
@pytest.mark.parametrize("kahan", [False, True])
def test_small_image_prior_updates_bit_for_bit(lm, n, kahan):
    """One event (its samples lie in different voxels) and prior updates alone:
    no sum depends on an order."""
    geo, ev = frame(lm, n, 1)
    pe = lm.event_setup(geo, ev, 1)
    rng = np.random.default_rng(1)
    sens = torch.from_numpy(rng.uniform(1, 2, geo.V).astype(np.float32)).cuda()
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, geo.V).astype(np.float32)).cuda()
    out = []
    for kernel in (0, 1):
        st = lm.LMSPDHG(geo, pe, sens, x0, beta=0.02, n_subsets=1, knorm=H.knorm_closed(n), image_kernel=kernel, kahan=kahan,
                        group=16)
        st.updates([1] * 5)
        out.append([t.cpu().numpy() for t in (st.x(), st.z(), st.w())])
        st.close()
    assert np.abs(out[0][2]).max() > 0
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
