"""GPU parity of the linear adjoint's warp-per-pair kernel (2D, straight legs)
at the sizes where it can go wrong, against the oracle's adjoint: in band
(|nu| <= 1/4, the echoes' band) to the FP32 path's 1e-4, over the full band to
1e-3 (the cubic Farrow form's weight error), as the other adjoint tests."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, in_band, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,dx,dy,x0,y0,P,C", [
    (64, 64, 0.015, 0.015, 2.0, 20.0, 9, 3),       # one whole tile
    (1, 1, 0.02, 0.02, 2.0, 20.0, 3, 1),           # one pixel, one pair a ping
    (65, 31, 0.02, 0.015, 2.0, 20.0, 5, 2),        # one pixel into the next tile, half lines
    (130, 97, 0.015, -0.02, 0.0, 22.0, 11, 4),     # ragged, backwards along y
    (70, 66, 0.02, 0.02, 16.0, 12.0, 7, 2),        # squinted: lanes along x
    (80, 50, 0.004, 0.004, 2.0, 20.0, 6, 3),       # lanes closer than a half sample: rows shared
    (90, 70, 0.02, 0.02, -0.5, -0.6, 8, 2),        # under the track: near pairs, no common direction
    (40, 70, 0.045, 0.045, 1.0, 20.0, 4, 2)])      # near the coarsest spacing taken: the longest rows
def test_adjoint_2d(nx, ny, dx, dy, x0, y0, P, C):
    g = synth.Grid(x0, y0, 0.0, dx, dy, 0.0, nx, ny, 1)
    w = synth.workload("small_2d", grid=g, n_pings=P, n_rx=C, n_samples=1024, t0=0.008 if y0 < 15 else 0.025,
                       altitude=10.0)
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    img = synth.random_image((1, ny, nx), seed=61).astype(np.complex64)
    out = torch.empty((P, C, 1024), dtype=torch.complex64, device="cuda")
    sas.sas_backproject_adjoint(geom.h, sas.grid_from(g), sas.kaiser(4.0), torch.from_numpy(img).cuda(), out)
    geom.sync_status()
    geom.close()
    tx, rx = oracle_positions(nav)
    ref = oracle.backproject_adjoint(tx, rx, oracle_signal(w), img.reshape(-1), 8, 4.0, grid_pixels(g))
    got = out.cpu().numpy()
    assert np.abs(ref).max() > 0
    assert oracle.rel_l2(in_band(got), in_band(ref)) < 1e-4
    assert oracle.rel_l2(got, ref) < 1e-3
