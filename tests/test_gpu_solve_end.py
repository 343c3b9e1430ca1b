"""Where the solve of Eq. 8 ends: at the minimum, also where its steps shrink slowly."""
import numpy as np
import pytest

import paper_2101_05888_gb300 as sas
from oracle import micronav as mn

import _dpc
from test_gpu_micronav import C_SOUND, _Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("huber,outliers,size,lam,P", [
    (0.0, 0.0, 0.0, 1e-3, 16),          # squares: the steps shrink a hundredfold each
    (2e-5, 0.1, 4e-6, 1e-3, 16),        # a threshold below the noise: a third each
    (2e-5, 0.1, 4e-6, 1e-3, 40),
    (1e-5, 0.2, 4e-4, 1e-3, 16)])       # large outliers
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_a_second_solve_stays(seed, huber, outliers, size, lam, P):
    """A solve from the solution, with the damping of a first trial again, does not move it:
    nodes (10 m) round at 2e-15 of their value and their steps end near 1e-12 m, which is
    2e-11 m/s over the 50 ms ping interval; a hundred times that is allowed.  Two evaluations of
    the loss differ by its rounding, up to 1e-11 each."""
    rng = np.random.default_rng(seed)
    pl = _dpc.platform(P=P, seed=seed)
    vy, vz = _dpc.true_velocities(P, seed=seed + 1)
    meas = _dpc.measurements(pl, 6, 0.025, 0.05, 2)
    ps = mn.footprints(pl, np.zeros(P), np.zeros(P), meas, C_SOUND)
    meas.delay = mn.model_delays(pl, vy, vz, meas, ps, C_SOUND) + rng.normal(0, 5e-8, meas.ping.size)
    if outliers:
        bad = rng.choice(meas.delay.size, int(meas.delay.size * outliers), replace=False)
        meas.delay[bad] += size * rng.choice([-1, 1], bad.size)
    meas.weight = rng.uniform(0.5, 1.0, meas.ping.size)
    z_dvl = mn.heave_positions(pl, vz) + rng.normal(0, 0.002, P)
    prob = _Problem(pl, meas, z_dvl, lam, 10 * lam, huber=huber, ps=ps)
    gy, gz = (torch.zeros(P, dtype=torch.float64, device="cuda") for _ in range(2))
    loss, iters = sas.sas_dpc_solve(prob.pr, gy, gz, 2000)
    hy, hz = gy.clone(), gz.clone()
    loss2, _ = sas.sas_dpc_solve(prob.pr, hy, hz, 2000)
    moved = max(float((hy - gy).abs().max()), float((hz - gz).abs().max()))
    print("huber %g P %d: %d steps, moved %.1e m/s, loss %.3e" % (huber, P, iters, moved, (loss2 - loss) / loss))
    assert moved < 2e-9
    assert abs(loss2 - loss) <= 2e-11 * loss
