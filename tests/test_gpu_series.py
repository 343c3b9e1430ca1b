"""GPU parity of the column series (forward pass, straight legs) where it can
go wrong: pairs on both sides of the range from which it holds, grids that run
backwards along the column's axis, beam edges on near pairs.

Tolerance: the FP32 path's 1e-4 (relative complex L2) of the other forward
tests: the Farrow form's 3.7e-5, FP32 phases 2e-5, the series' own 5e-6 rad."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BETA = 4.0


def _compare(w, store=sas.SAS_ECHO_C64, tol=1e-4):
    nav = synth.nav(w)
    echo = synth.random_echo(w.n_pings, w.n_rx, w.n_samples, seed=51)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.upload_echo(echo, store)
    img = geom.backproject(sas.grid_from(w.grid), sas.kaiser(BETA)).cpu().numpy()
    geom.sync_status()
    stored = geom.download_echo().cpu().numpy()
    geom.close()
    tx, rx = oracle_positions(nav)
    ref = oracle.backproject(tx, rx, oracle_signal(w), stored, 8, BETA, grid_pixels(w.grid)).reshape(img.shape)
    assert oracle.rel_l2(img, ref) < tol


@pytest.mark.parametrize("y0,dy,alt", [(0.5, 0.015, 2.0),      # every pair nearer than the series' range
                                       (5.0, 0.02, 4.0),       # both kinds within a tile's pairs
                                       (9.0, -0.015, 2.0),     # slots run towards the track
                                       (40.0, -0.02, 10.0)])   # far: the series everywhere
def test_2d_near_and_far(y0, dy, alt):
    g = synth.Grid(-0.4, y0, 0.0, 0.015, dy, 0.0, 61, 150, 1)
    w = synth.workload("small_2d", grid=g, n_pings=80, n_rx=3, n_samples=1024, t0=0.0 if y0 < 20 else 0.05,
                       altitude=alt)
    _compare(w)


@pytest.mark.parametrize("z0,dz", [(-1.2, 0.02), (0.3, -0.02)])
@pytest.mark.parametrize("store,tol", [(sas.SAS_ECHO_C64, 1e-4), (sas.SAS_ECHO_C32_F16, 1e-3)])
def test_3d_near_and_far(z0, dz, store, tol):
    """Layers from 0.8 m below the sensors: columns on both sides of the
    series' 2 m, seen obliquely by the far pings of the lattice."""
    g = synth.Grid(0.1, 0.2, z0, 0.02, 0.02, dz, 21, 33, 19)
    w = synth.workload("volume_3d", grid=g, n_pings=25, n_rx=4, n_samples=1024, lattice=5, lattice_pitch=0.9,
                       echo_dtype="c64")
    _compare(w, store, tol)


def test_beam_edge_on_near_pairs():
    """Per-pixel beam tests in the exact form; pixels with ambiguous terms are
    left out."""
    g = synth.Grid(0.0, 2.0, 0.0, 0.02, 0.02, 0.0, 112, 96, 1)
    w = synth.workload("small_2d", grid=g, n_pings=40, n_rx=2, n_samples=1024, t0=0.0, altitude=3.0)
    nav = synth.nav(w)
    width = np.deg2rad(25.0)
    echo = synth.random_echo(w.n_pings, w.n_rx, w.n_samples, seed=52)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.set_beam(width, 1)
    geom.upload_echo(echo)
    img = geom.backproject(sas.grid_from(w.grid), sas.kaiser(BETA)).cpu().numpy().reshape(-1)
    geom.sync_status()
    geom.close()
    tx, rx = oracle_positions(nav)
    sure, amb = oracle.backproject_beam_split(tx, rx, oracle_signal(w), echo, 8, BETA, grid_pixels(w.grid),
                                              nav["att"], width, 1, eps=2e-6)
    clean = amb == 0.0
    assert clean.mean() > 0.98
    assert oracle.rel_l2(img[clean], sure[clean]) < 1e-4
