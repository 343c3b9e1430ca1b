"""Forward images whose tiles are split over several CTAs: the parts are added in
a fixed order, so two runs agree bit for bit, with and without accumulation; and
the solve of Eq. 8 over sizes that take one to four reductions."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth
from oracle import micronav as mn

import _dpc
from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal
from test_gpu_micronav import C_SOUND, _Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,px,P,C,store,tol", [
    (256, 100, 0.02, 61, 3, sas.SAS_ECHO_C64, 1e-4),         # two Farrow buffers, uneven splits
    (57, 33, 0.015, 150, 1, sas.SAS_ECHO_C64, 1e-4),         # four tiles, many splits
    (900, 600, 0.015, 9, 2, sas.SAS_ECHO_C32_BF16, 1e-3)])   # more tiles than CTAs in a wave
def test_split_images_are_reproducible(nx, ny, px, P, C, store, tol):
    g = synth.Grid(1.0, 20.0, 0.0, px, px, 0.0, nx, ny, 1)
    w = synth.workload("small_2d", grid=g, n_pings=P, n_rx=C, n_samples=1024, t0=0.025)
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.upload_echo(synth.random_echo(P, C, 1024, seed=71), store)
    stored = geom.download_echo().cpu().numpy()
    a = geom.backproject(sas.grid_from(g), sas.kaiser(4.0))
    b = geom.backproject(sas.grid_from(g), sas.kaiser(4.0))
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    geom.backproject(sas.grid_from(g), sas.kaiser(4.0), image=b, accumulate=True)
    geom.sync_status()
    geom.close()
    assert oracle.rel_l2(b.cpu().numpy(), 2.0 * a.cpu().numpy()) < 1e-6      # one more FP32 rounding
    tx, rx = oracle_positions(nav)
    pix = grid_pixels(g)
    keep = np.random.default_rng(7).permutation(len(pix))[:4000]
    ref = oracle.backproject(tx, rx, oracle_signal(w), stored, 8, 4.0, pix[keep])
    assert oracle.rel_l2(a.cpu().numpy().reshape(-1)[keep], ref) < tol


@pytest.mark.parametrize("P,chunk", [(2, 0), (4, 8), (5, 0), (33, 0), (70, 0), (70, 16)])
def test_solve_sizes(P, chunk):
    """n = 2 P unknowns: less than a block of 8, one segment, several, two systems
    (chunk 16: segments of two blocks, four systems); the oracle's minimum."""
    pl = _dpc.platform(P=P)
    vy, vz = _dpc.true_velocities(P, seed=P)
    meas = _dpc.measurements(pl, 6, 0.025, 0.05, 2)
    ps = mn.footprints(pl, np.zeros(P), np.zeros(P), meas, C_SOUND)
    meas.delay = mn.model_delays(pl, vy, vz, meas, ps, C_SOUND)
    z_dvl = mn.heave_positions(pl, vz)
    lam1, lam2 = 1e-3, 1e-2
    ry, rz, rloss = mn.solve(pl, np.zeros(P), np.zeros(P), meas, ps, C_SOUND, z_dvl, lam1, lam2)
    prob = _Problem(pl, meas, z_dvl, lam1, lam2, ps=ps)
    gy, gz = (torch.zeros(P, dtype=torch.float64, device="cuda") for _ in range(2))
    sas.sas_debug_dpc_solve_chunk(chunk)
    try:
        loss, _ = sas.sas_dpc_solve(prob.pr, gy, gz, 200)
    finally:
        sas.sas_debug_dpc_solve_chunk(0)
    gy, gz = gy.cpu().numpy(), gz.cpu().numpy()
    # the oracle's loss to 1e-9 and velocities to 1e-6 m/s of 3e-2, as for the other solves
    assert abs(mn.total_loss(pl, gy, gz, meas, ps, C_SOUND, z_dvl, lam1, lam2) - rloss) <= 1e-9 * rloss + 1e-20
    assert np.abs(gy - ry).max() < 1e-6 and np.abs(gz - rz).max() < 1e-6
