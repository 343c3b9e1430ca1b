"""The column series of the forward pass, which 16-bit echoes over straight legs take: pairs
on both sides of the range from which it holds, slots that run backwards, beam edges, 2D
and 3D.

The reference is the image by FP64 geometry from the stored echo with the quadratic taps the
kernel applies (their three coefficients a half and tap, recovered from
sas_interp_eval_form), so the quadratic's own interpolation error drops out and what is
left is the kernel's arithmetic: FP32 phases and paths 2e-5, the series' 5e-6 rad, and 1e-5
from pixels whose fraction falls on the other side of a half: 1e-4, as the FP32 path's other
tests.  A wrong cubic term is 1e-2 rad, a wrong quartic one up to 9e-4 rad, at the near ranges."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BETA, TOL = 4.0, 1e-4
STORES = [sas.SAS_ECHO_C32_F16, sas.SAS_ECHO_C32_BF16]


def _quadratic_taps():
    """[2][8][3]: the coefficients (highest power first) in g = frac(2u) - 1/2 of every half and tap."""
    g = np.array([-0.4375, 0.0, 0.4375])
    f = np.concatenate([(g + 0.5) / 2, (g + 1.5) / 2]).astype(np.float32)
    out = torch.empty((6, 8), device="cuda")
    sas.sas_interp_eval_form(sas.kaiser(BETA), 2, torch.from_numpy(f).cuda(), 6, out)
    w = out.double().cpu().numpy()
    return np.stack([np.polyfit(g, w[3 * h:3 * h + 3], 2).T for h in range(2)])


def _reference(tx, rx, sig, echo, pix, att=None, width=0.0, side=1, eps=2e-6):
    """The image at pix, and which pixels have a beam decision within eps of an edge."""
    taps = _quadratic_taps()
    P, C, Ns = echo.shape
    e = np.zeros((P, C, Ns + 16), complex)
    e[:, :, 8:8 + Ns] = echo
    img, amb = np.zeros(len(pix), complex), np.zeros(len(pix), bool)
    k = np.tan(0.5 * width)

    def sees(i, s):
        b = (pix - s) @ oracle.attitude_matrix(*att[i])
        m = np.abs(b[:, 0]) - k * side * b[:, 1]
        return m <= 0.0, np.abs(m) <= eps * (np.abs(b[:, 0]) + np.abs(b[:, 1]))

    for i in range(P):
        dT = np.linalg.norm(pix - tx[i], axis=1)
        st, at = sees(i, tx[i]) if width else (True, False)
        for c in range(C):
            tau = (dT + np.linalg.norm(pix - rx[i, c], axis=1)) / sig.c
            u = (tau - sig.t0) * sig.fs
            n = np.floor(u)
            h = (u - n >= 0.5).astype(int)
            g = 2.0 * (u - n) - h - 0.5
            w = (taps[h, :, 0] * g[:, None] + taps[h, :, 1]) * g[:, None] + taps[h, :, 2]
            at_ = np.clip(n.astype(int), -5, Ns + 3)[:, None] + np.arange(-3, 5) + 8
            v = np.sum(w * e[i, c][np.clip(at_, 0, Ns + 15)], axis=1) * np.exp(2j * np.pi * sig.fc * tau)
            if width:
                sr, ar = sees(i, rx[i, c])
                v = np.where(st & sr, v, 0.0)
                amb |= at | ar
            img += v
    return img, amb


def _compare(w, store, width=0.0):
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    if width:
        geom.set_beam(width, 1)
    geom.upload_echo(synth.random_echo(w.n_pings, w.n_rx, w.n_samples, seed=51), store)
    img = geom.backproject(sas.grid_from(w.grid), sas.kaiser(BETA)).cpu().numpy().reshape(-1)
    geom.sync_status()
    stored = geom.download_echo().cpu().numpy().astype(complex)
    geom.close()
    tx, rx = oracle_positions(nav)
    ref, amb = _reference(tx, rx, oracle_signal(w), stored, grid_pixels(w.grid), nav["att"], width)
    assert np.mean(~amb) > 0.98
    err = oracle.rel_l2(img[~amb], ref[~amb])
    print("%.2e" % err)
    assert err < TOL


@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("y0,dy,alt,P", [(0.5, 0.015, 2.0, 40),      # every pair nearer than the series' range
                                         (5.0, 0.02, 4.0, 80),       # both kinds within a tile's pairs
                                         (9.0, -0.015, 2.0, 40),     # slots run towards the track
                                         (40.0, -0.02, 10.0, 40),    # far: the series everywhere
                                         (40.0, 0.02, 10.0, 1)])     # one ping: unsplit
def test_2d(y0, dy, alt, P, store):
    g = synth.Grid(-0.4, y0, 0.0, 0.015, dy, 0.0, 61, 100, 1)
    _compare(synth.workload("small_2d", grid=g, n_pings=P, n_rx=3, n_samples=1024, t0=0.0 if y0 < 20 else 0.05,
                            altitude=alt), store)


@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("z0,dz", [(-1.2, 0.02), (0.3, -0.02)])
def test_3d(z0, dz, store):
    g = synth.Grid(0.1, 0.2, z0, 0.02, 0.02, dz, 21, 33, 19)
    _compare(synth.workload("volume_3d", grid=g, n_pings=25, n_rx=4, n_samples=1024, lattice=5, lattice_pitch=0.9),
             store)


@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("y0,alt,width", [(2.0, 3.0, 25.0),          # near: the exact form under the beam test
                                          (12.0, 3.0, 20.0)])        # far: the series under it
def test_beam_edges(y0, alt, width, store):
    g = synth.Grid(0.0, y0, 0.0, 0.02, 0.02, 0.0, 112, 96, 1)
    _compare(synth.workload("small_2d", grid=g, n_pings=40, n_rx=2, n_samples=1024, t0=0.0, altitude=alt), store,
             np.deg2rad(width))
