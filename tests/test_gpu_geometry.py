"""Sensor positions over the shapes of the geometry kernel's blocks (8 or 32 pings, 128 threads):
part of a block, many blocks, more sensors than threads; and that many pings cost no more
than one thread a ping would take."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _geom(P, C, seed=3):
    rng = np.random.default_rng(seed)
    pos, att = rng.normal(0, 50, (P, 3)), rng.normal(0, 1, (P, 3))
    tx, rx = rng.normal(0, 1, 3), rng.normal(0, 1, (C, 3))
    return pos, att, tx, rx, sas.Geometry(pos, att, tx, rx, sas.make_signal(100e3, 40e3, 1500.0, 0.0, 64))


@pytest.mark.parametrize("P,C", [(1, 1), (7, 15), (8, 16), (9, 1), (3, 200), (1, 2000), (257, 5), (8191, 2), (8200, 3)])
def test_positions_match_oracle(P, C):
    pos, att, tx, rx, geom = _geom(P, C)
    off = np.random.default_rng(4).normal(0, 0.1, (P, 3))
    geom.set_offsets(off)
    gtx, grx = geom.positions()
    rtx, rrx = oracle.sensor_positions(pos, att, tx, rx, off)
    geom.close()
    # FP64 throughout: 1e-12 m of 200 m
    assert np.abs(gtx.cpu().numpy() - rtx).max() < 1e-12
    assert np.abs(grx.cpu().numpy() - rrx).max() < 1e-12


def test_moving_many_pings_is_fast():
    """50000 pings x 8 receivers write 22 MB; a warp a ping took 215 us on the FP64 pipe, a
    thread a ping 43 us."""
    *_, geom = _geom(50000, 8)
    off = torch.zeros((50000, 3), dtype=torch.float64, device="cuda")
    for _ in range(3):
        geom.set_offsets(off)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(20):
        geom.set_offsets(off)
    b.record()
    torch.cuda.synchronize()
    geom.close()
    assert a.elapsed_time(b) / 20 < 0.1
