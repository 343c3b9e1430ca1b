"""The reference terms of receiver motion away from a survey's few metres a second: fast
platforms (|v| / c up to 0.05) and receivers exactly at an image tile's centre."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("speed", [6.0, 75.0, 150.0])
def test_fast_receivers(speed):
    """Grids of 8 x 8 micrometre pixels: the differential path D stays below 6.4e-5 m, so the
    pixel correction D / (1 + eps), expanded to eps^2, is off by eps^3 D <= 6.4e-8 m
    (3e-5 rad at |v| / c = 0.1) and the image shows the reference terms; the FP32 path's 1e-4
    of the other forward tests.  Twelve grids, as the pixels of one are alike."""
    w = synth.workload("stripmap_2d", grid=synth.Grid(0.0, 40.0, 0.0, 1e-6, 1e-6, 0.0, 8, 8, 1), n_pings=24, n_rx=3,
                       n_samples=4096, t0=0.05)
    nav = synth.nav(w)
    vel = np.tile(speed * np.array([0.8, 0.55, -0.24]), (24, 1))
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.set_velocity(vel)
    echo = synth.random_echo(24, 3, 4096, seed=101)
    geom.upload_echo(echo)
    tx, rx = oracle_positions(nav)
    got, ref = [], []
    for k in range(12):
        g = synth.Grid(0.3 * k, 40.0 + 1.7 * k, 0.0, 1e-6, 1e-6, 0.0, 8, 8, 1)
        got.append(geom.backproject(sas.grid_from(g), sas.kaiser(4.0)).cpu().numpy().reshape(-1))
        ref.append(oracle.backproject(tx, rx, oracle_signal(w), echo, 8, 4.0, grid_pixels(g), vel=vel))
    geom.sync_status()
    geom.close()
    err = oracle.rel_l2(np.concatenate(got), np.concatenate(ref))
    print("speed %g: %.2e" % (speed, err))
    assert err < 1e-4


@pytest.mark.parametrize("moving", [True, False])
def test_receiver_at_a_tile_centre(moving):
    """The receiver of one ping at the centre of the first tile (56 x 32 pixels, between
    pixels), the transmitter 5 m behind it: finite, and the oracle's image."""
    px = 0.02
    g = synth.Grid(0.0, 0.0, 0.0, px, px, 0.0, 56, 32, 1)
    centre = np.array([27.5 * px, 15.5 * px, 0.0])
    tx_lever, rx_lever = np.array([-5.0, 0.0, 0.0]), np.zeros((1, 3))
    sig = sas.make_signal(synth.FC, synth.FS, synth.C_SOUND, 0.0, 512)
    geom = sas.Geometry(centre[None], np.zeros((1, 3)), tx_lever, rx_lever, sig)
    vel = np.array([[1.5, 0.3, -0.1]])
    if moving:
        geom.set_velocity(vel)
    echo = synth.random_echo(1, 1, 512, seed=102)
    geom.upload_echo(echo)
    img = geom.backproject(sas.grid_from(g), sas.kaiser(4.0)).cpu().numpy()
    geom.sync_status()
    geom.close()
    assert np.all(np.isfinite(img.view(np.float32)))
    pix = grid_pixels(g)
    ref = oracle.backproject((centre + tx_lever)[None], centre[None, None], oracle.Signal(
        synth.FC, synth.FS, synth.C_SOUND, 0.0, 512), echo, 8, 4.0, pix, vel=vel if moving else None).reshape(img.shape)
    # the receiver has moved 5 mm when the echo arrives, and the pixel correction is of
    # first order in that against the range: pixels beyond 0.2 m, to 0.42 rad x (5e-3 / 0.2)^2
    far = np.linalg.norm(pix - centre, axis=1).reshape(img.shape) > 0.2
    assert oracle.rel_l2(img[far], ref[far]) < 3e-4


@pytest.mark.parametrize("speed", [1.95, 60.0])
def test_adjoint_takes_the_forward_terms_with_beam_and_motion(speed):
    """<B e, G> = <e, B^H G> over a grid that beam edges sweep across: both passes form
    the same reference terms, so they take the same decisions and delays (one term
    decided differently moves the product by about 1; FP32 rounding by ~1e-6 of a random
    inner product's size, as in the dot test of the beam alone)."""
    g = synth.Grid(8.0, 40.0, 0.0, 0.03, 0.03, 0.0, 160, 60, 1)
    w = synth.workload("stripmap_2d", grid=g, n_pings=40, n_rx=2, n_samples=4096, t0=0.05)
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.set_beam(np.deg2rad(25.0), 1)
    geom.set_velocity(np.tile(speed * np.array([1.0, 0.02, -0.01]), (40, 1)))
    echo = synth.random_echo(40, 2, 4096, seed=103)
    geom.upload_echo(echo)
    G = synth.random_image((1, g.ny, g.nx), seed=104).astype(np.complex64)
    eadj = torch.empty((40, 2, 4096), dtype=torch.complex64, device="cuda")
    Be = geom.backproject(sas.grid_from(g), sas.kaiser(4.0)).cpu().numpy().reshape(-1).astype(np.complex128)
    sas.sas_backproject_adjoint(geom.h, sas.grid_from(g), sas.kaiser(4.0), torch.from_numpy(G).cuda(), eadj)
    geom.sync_status()
    geom.close()
    Gv = G.reshape(-1).astype(np.complex128)
    lhs = np.vdot(Be, Gv)
    rhs = np.vdot(echo.reshape(-1).astype(np.complex128), eadj.cpu().numpy().reshape(-1).astype(np.complex128))
    print("speed %g: %.2e" % (speed, abs(lhs - rhs) / (np.linalg.norm(Be) * np.linalg.norm(Gv) / np.sqrt(Gv.size))))
    assert abs(lhs - rhs) <= 2e-5 * np.linalg.norm(Be) * np.linalg.norm(Gv) / np.sqrt(Gv.size)
