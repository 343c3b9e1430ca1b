"""The time-varying gain where its scratch cannot be had: the device's stream-ordered
allocator is replaced, in a child process, by a pool of a few MB, so that the larger
allocation is refused without any memory being used up."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys
import torch
import paper_2101_05888_gb300 as sas

class Loc(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("id", ctypes.c_int)]

class Props(ctypes.Structure):
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("location", Loc),
                ("win32", ctypes.c_void_p), ("maxSize", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]

rows, n = int(sys.argv[1]), int(sys.argv[2])
g = torch.Generator(device="cuda"); g.manual_seed(5)
x = torch.view_as_complex(torch.randn((rows, n, 2), device="cuda", generator=g))
def run(with_outputs):
    out = torch.empty_like(x)
    med = torch.empty(n, dtype=torch.float64, device="cuda") if with_outputs else None
    gain = torch.empty(n, device="cuda") if with_outputs else None
    sas.sas_tvg(x, out, rows, n, 0.3, gain, med)
    torch.cuda.synchronize()
    return out, med, gain
a, b = run(True), run(False)
cu = ctypes.CDLL("libcuda.so.1")
pool, dev = ctypes.c_void_p(), torch.cuda.current_device()
props = Props(1, 0, Loc(1, dev), None, 4 << 20, 0)       # pinned, on this device, 4 MB at most
if cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) != 0 or cu.cuDeviceSetMemPool(dev, pool) != 0:
    sys.exit(77)
p = ctypes.c_void_p()
big = 4 * n * 2048
if cu.cuMemAllocFromPoolAsync(ctypes.byref(p), ctypes.c_size_t(big), pool, None) == 0:
    sys.exit(77)                                          # the driver does not hold the pool to its size
c, d = run(True), run(False)
bits = lambda t: torch.view_as_real(t)
assert torch.equal(bits(a[0]), bits(c[0])) and torch.equal(bits(b[0]), bits(d[0])) and torch.equal(bits(a[0]), bits(b[0]))
assert torch.equal(a[1], c[1]) and torch.equal(a[2], c[2])
"""


@pytest.mark.parametrize("rows,n", [(9001, 8192), (20000, 8192)])
def test_gain_without_scratch(rows, n):
    r = subprocess.run([sys.executable, "-c", CHILD, str(rows), str(n)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    if r.returncode == 77:
        pytest.skip("no pool of a bounded size here")
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("rows,n", [(12287, 9), (12288, 9), (8191, 2048), (8192, 2048), (20000, 5), (32767, 5)])
def test_select_on_both_sides_of_its_rules(rows, n):
    """Row counts and widths around the lines of the bracketed select, and columns whose
    bracket holds more rows than the scratch has room for (half of them equal)."""
    import paper_2101_05888_gb300 as sas
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + n)
    x = torch.view_as_complex(torch.randn((rows, n, 2), device="cuda", generator=g))
    x[:, 1] = 0.25 + 0.5j
    x[::2, 2] = 0.75j                                   # half the rows equal, near the median
    x[:, 3] = torch.linspace(0.1, 2.0, rows, device="cuda")
    out, med = torch.empty_like(x), torch.empty(n, dtype=torch.float64, device="cuda")
    sas.sas_tvg(x, out, rows, n, 0.3, None, med)
    # re*re + im*im rounded to FP32
    v = torch.view_as_real(x)
    p = torch.sort(v[..., 0] * v[..., 0] + v[..., 1] * v[..., 1], dim=0).values.double()
    ref = 0.5 * (p[(rows - 1) // 2] + p[rows // 2])
    # PyTorch may fuse the sum (at most one unit in the last place of FP32)
    assert bool(((med - ref).abs() <= 1.2e-7 * ref).all())
