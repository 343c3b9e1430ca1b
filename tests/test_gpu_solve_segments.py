"""The solve of Eq. 8 by segments of two, four and eight blocks over a track that takes
three systems at eight (75 blocks of unknowns, then 10, then 2)."""
import numpy as np
import pytest

import paper_2101_05888_gb300 as sas
from oracle import micronav as mn

import _dpc
from test_gpu_micronav import C_SOUND, _Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_segments_of_a_long_track():
    P = 300
    rng = np.random.default_rng(5)
    pl = _dpc.platform(P=P)
    vy, vz = _dpc.true_velocities(P, seed=6)
    meas = _dpc.measurements(pl, 2, 0.03, 0.05, 2)
    ps = mn.footprints(pl, np.zeros(P), np.zeros(P), meas, C_SOUND)
    meas.delay = mn.model_delays(pl, vy, vz, meas, ps, C_SOUND) + rng.normal(0, 5e-8, meas.ping.size)
    z_dvl = mn.heave_positions(pl, vz) + rng.normal(0, 0.002, P)
    lam = (1e-3, 1e-2)
    prob = _Problem(pl, meas, z_dvl, *lam, ps=ps)
    got = {}
    for rows in (0, 16, 32, 64):                      # segments of 8, 2, 4 and 8 blocks
        gy, gz = (torch.zeros(P, dtype=torch.float64, device="cuda") for _ in range(2))
        sas.sas_debug_dpc_solve_chunk(rows)
        try:
            _, iters = sas.sas_dpc_solve(prob.pr, gy, gz, 200)
        finally:
            sas.sas_debug_dpc_solve_chunk(0)
        got[rows] = (gy.cpu().numpy(), gz.cpu().numpy(), iters)
    for rows in (16, 32, 64):
        # one minimum (the bound of a second solve), by steps as good as each other's
        assert np.abs(got[rows][0] - got[0][0]).max() < 2e-9 and np.abs(got[rows][1] - got[0][1]).max() < 2e-9
        assert abs(got[rows][2] - got[0][2]) <= 3
    # the oracle's loss is stationary there: the Newton step along any direction is below
    # 1e-6 m/s, the bound of the other solves (differences at 1e-3 m/s, where the loss is
    # quadratic to 1e-6 and moves by far more than it rounds)
    y, z, _ = got[0]
    loss = lambda a, b: mn.total_loss(pl, a, b, meas, ps, C_SOUND, z_dvl, *lam)
    l0, h = loss(y, z), 1e-3
    for _ in range(3):
        d = rng.choice([-1.0, 1.0], (2, P))
        up, dn = loss(y + h * d[0], z + h * d[1]), loss(y - h * d[0], z - h * d[1])
        assert up > l0 and dn > l0
        assert abs(up - dn) / (2 * h) <= 1e-6 * (up + dn - 2 * l0) / (h * h)
