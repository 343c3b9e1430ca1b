"""Small images of many pings: the parts' sum at many parts, and what choosing the parts
costs the host."""
import time

import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _geom(P, C):
    g = synth.Grid(0.0, 20.0, 0.0, 0.015, 0.015, 0.0, 33, 21, 1)
    w = synth.workload("small_2d", grid=g, n_pings=P, n_rx=C, n_samples=512, t0=0.025, ping_spacing=4.0 / P)
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.upload_echo(synth.random_echo(P, C, 512, seed=P))
    return w, nav, geom


@pytest.mark.parametrize("P,C", [(13, 8), (15, 8), (16, 8), (17, 8), (47, 4), (300, 3)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_sums_of_many_parts(P, C, accumulate):
    """One tile: a part a ping, from a few (a thread a pixel) to 300 (eight threads a pixel)."""
    w, nav, geom = _geom(P, C)
    img = torch.full((1, 21, 33), 2.0 - 1.0j, dtype=torch.complex64, device="cuda")
    geom.backproject(sas.grid_from(w.grid), sas.kaiser(4.0), image=img, accumulate=accumulate)
    geom.sync_status()
    echo = geom.download_echo().cpu().numpy()
    geom.close()
    tx, rx = oracle_positions(nav)
    ref = oracle.backproject(tx, rx, oracle_signal(w), echo, 8, 4.0, grid_pixels(w.grid)).reshape(img.shape)
    got = img.cpu().numpy() - (2.0 - 1.0j if accumulate else 0.0)
    assert oracle.rel_l2(got, ref) < 1e-4


def test_many_pings_cost_the_host_no_more():
    """The host's part of a call over 5000 pings stays near that over 64 (trying every split,
    one after the other, made it 3.5 times as long)."""
    med = {}
    for P in (64, 5000):
        w, _, geom = _geom(P, 1)
        grid, k = sas.grid_from(w.grid), sas.kaiser(4.0)
        img = torch.empty((1, 21, 33), dtype=torch.complex64, device="cuda")
        t = []
        for _ in range(300):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            geom.backproject(grid, k, image=img)
            t.append(time.perf_counter() - t0)
        torch.cuda.synchronize()
        geom.close()
        med[P] = np.median(t[50:])
    assert med[5000] < 2.0 * med[64]
