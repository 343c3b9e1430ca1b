"""Images and offset gradients recorded in a CUDA graph: the graph owns the scratch of
its calls, so calls of the same handle that need larger scratch, made between the
capture and a replay, leave it alone."""
import numpy as np
import pytest

import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import synth

from _scene import lib_signal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _handle():
    g = synth.Grid(1.0, 20.0, 0.0, 0.015, 0.015, 0.0, 60, 50, 1)
    w = synth.workload("small_2d", grid=g, n_pings=48, n_rx=4, n_samples=1024, t0=0.025)
    geom = sas.Geometry.from_nav(synth.nav(w), lib_signal(w))
    geom.upload_echo(synth.random_echo(48, 4, 1024, seed=91))
    return geom, sas.grid_from(g)


def _image(grid, seed):
    return torch.from_numpy(synth.random_image((1, grid.ny, grid.nx), seed=seed).astype(np.complex64)).cuda()


def test_captured_gradient_and_image_survive_larger_calls():
    geom, small = _handle()
    k = sas.kaiser(4.0)
    large = sas.make_grid(small.x0, small.y0, 0.0, 0.015, 0.015, 0.0, 900, 700)
    gimg = _image(small, 92)
    img = torch.empty((1, small.ny, small.nx), dtype=torch.complex64, device="cuda")
    grad = torch.empty((48, 3), dtype=torch.float64, device="cuda")
    geom.backproject(small, k, image=img)                      # as in plain calls
    sas.sas_backproject_adjoint(geom.h, small, k, gimg, None, grad)
    img0, grad0 = img.clone(), grad.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        geom.backproject(small, k, image=img)
        sas.sas_backproject_adjoint(geom.h, small, k, gimg, None, grad)
    for _ in range(2):
        # larger scratch for both calls; then other allocations, which would take what they freed
        big = geom.backproject(large, k)
        big_grad = torch.empty_like(grad)
        sas.sas_backproject_adjoint(geom.h, large, k, _image(large, 93), None, big_grad)
        torch.cuda.synchronize()
        hold = [torch.full((1 << 22,), 7.0, device="cuda") for _ in range(8)]
        big0, big_grad0 = big.clone(), big_grad.clone()
        img.zero_()
        grad.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(img), torch.view_as_real(img0))
        assert torch.equal(grad, grad0)
        assert all(bool((h == 7.0).all()) for h in hold)
        again = geom.backproject(large, k)
        sas.sas_backproject_adjoint(geom.h, large, k, _image(large, 93), None, big_grad)
        assert torch.equal(torch.view_as_real(again), torch.view_as_real(big0)) and torch.equal(big_grad, big_grad0)
    geom.sync_status()
    geom.close()


@pytest.mark.parametrize("store", [sas.SAS_ECHO_C64, sas.SAS_ECHO_C32_BF16])
def test_images_allocate_nothing(store):
    """After the upload, images of growing size in plain calls (one part, many parts, a whole wave of
    tiles) leave the free device memory as it is."""
    geom, _ = _handle()
    geom.upload_echo(synth.random_echo(48, 4, 1024, seed=94), store)
    k = sas.kaiser(4.0)
    sizes = [(1, 1), (60, 50), (300, 200), (900, 700), (1500, 1100), (2000, 1500)]
    imgs = [torch.empty((1, ny, nx), dtype=torch.complex64, device="cuda") for nx, ny in sizes]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for (nx, ny), img in zip(sizes, imgs):
        geom.backproject(sas.make_grid(1.0, 20.0, 0.0, 0.015, 0.015, 0.0, nx, ny), k, image=img)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
    geom.sync_status()
    geom.close()
