"""The widest delay spans a tile may have: coarse pixels that the offset gradient of
16-bit echoes takes with two Farrow buffers, and the first ones that are refused."""
import numpy as np
import pytest

import oracle
import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import grid_pixels, lib_signal, oracle_positions, oracle_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(px, store):
    g = synth.Grid(1.0, 20.0, 0.0, px, px, 0.0, 70, 40, 1)
    w = synth.workload("small_2d", grid=g, n_pings=9, n_rx=2, n_samples=1024, t0=0.025)
    nav = synth.nav(w)
    geom = sas.Geometry.from_nav(nav, lib_signal(w))
    geom.upload_echo(synth.random_echo(9, 2, 1024, seed=81), store)
    img = synth.random_image((1, 40, 70), seed=82).astype(np.complex64)
    return w, nav, geom, img


@pytest.mark.parametrize("store", [sas.SAS_ECHO_C32_F16, sas.SAS_ECHO_C32_BF16])
@pytest.mark.parametrize("px", [0.0562, 0.0572, 0.0605])       # 97, 99 and 104 samples either way
def test_offset_gradient_of_coarse_pixels(px, store):
    w, nav, geom, img = _scene(px, store)
    stored = geom.download_echo().cpu().numpy()
    grad = torch.empty((9, 3), dtype=torch.float64, device="cuda")
    sas.sas_backproject_adjoint(geom.h, sas.grid_from(w.grid), sas.kaiser(4.0), torch.from_numpy(img).cuda(), None, grad)
    geom.sync_status()
    geom.close()
    tx, rx = oracle_positions(nav)
    ref = oracle.vjp_offsets(tx, rx, oracle_signal(w), stored, 8, 4.0, grid_pixels(w.grid), img.reshape(-1))
    assert oracle.rel_l2(grad.cpu().numpy(), ref) < 1e-3         # as the other offset gradients


@pytest.mark.parametrize("px,store,forward", [(0.0613, sas.SAS_ECHO_C32_F16, True),      # 106: only the image
                                              (0.0705, sas.SAS_ECHO_C32_F16, False),     # 121
                                              (0.0480, sas.SAS_ECHO_C64, False)])        # 83
def test_wider_spans_are_refused(px, store, forward):
    w, nav, geom, img = _scene(px, store)
    grid, grad = sas.grid_from(w.grid), torch.empty((9, 3), dtype=torch.float64, device="cuda")
    with pytest.raises(sas.SasError) as e:
        sas.sas_backproject_adjoint(geom.h, grid, sas.kaiser(4.0), torch.from_numpy(img).cuda(), None, grad)
    assert e.value.code == sas.SAS_ERR_UNSUPPORTED
    if forward:
        geom.backproject(grid, sas.kaiser(4.0))
    else:
        with pytest.raises(sas.SasError) as e:
            geom.backproject(grid, sas.kaiser(4.0))
        assert e.value.code == sas.SAS_ERR_UNSUPPORTED
    geom.sync_status()
    geom.close()
