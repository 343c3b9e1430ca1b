"""The conditioning kernels on both sides of their size rules: the bracketed select
of the TVG for middling row counts (exact medians whatever the sample says) and the
matched filter's block lengths."""
import numpy as np
import pytest

import oracle
from oracle import conditioning as cond
import paper_2101_05888_gb300 as sas

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n", [(8191, 9), (8192, 40), (9001, 33), (32767, 8)])
def test_tvg_row_rules(rows, n):
    rng = np.random.default_rng(rows)
    e = (rng.normal(size=(rows, n)) + 1j * rng.normal(size=(rows, n))).astype(np.complex64)
    e[:, 1] = 0.5 - 0.25j                                  # one value
    e[:, 2] = np.linspace(0.1, 2.0, rows)                  # ordered along the rows
    e[::8, 3] *= 50.0                                      # the sampled rows are not typical
    e[::4, 4] = 0.0
    d_in = torch.from_numpy(e).cuda()
    out, med = torch.empty_like(d_in), torch.empty(n, dtype=torch.float64, device="cuda")
    sas.sas_tvg(d_in, out, rows, n, 0.2, None, med)
    torch.cuda.synchronize()
    ref, _, P = cond.tvg(e, 0.2)
    assert np.array_equal(med.cpu().numpy(), P)            # exact selection
    assert oracle.rel_l2(out.cpu().numpy(), ref) < 1e-6


@pytest.mark.parametrize("n", [60, 1000, 5000])
@pytest.mark.parametrize("L", [50, 128, 129, 700, 2100])
def test_matched_filter_block_rule(n, L):
    rng = np.random.default_rng(n + L)
    raw = (rng.normal(size=(3, n)) + 1j * rng.normal(size=(3, n))).astype(np.complex64)
    rep = np.exp(1j * rng.uniform(0, 2 * np.pi, L)).astype(np.complex64)
    out = torch.empty((3, n), dtype=torch.complex64, device="cuda")
    sas.sas_matched_filter(torch.from_numpy(raw).cuda(), 3, n, torch.from_numpy(rep).cuda(), L, out)
    torch.cuda.synchronize()
    # the definition by FP64 transforms; FP32 transforms of up to 16384 points: 1e-5
    m = n + L
    r = rep.astype(np.complex128)
    ref = np.fft.ifft(np.fft.fft(raw.astype(np.complex128), m) * np.conj(np.fft.fft(r, m)))[:, :n] / np.sum(np.abs(r) ** 2)
    assert oracle.rel_l2(out.cpu().numpy(), ref) < 1e-5
