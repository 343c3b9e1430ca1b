"""The conditioning calls in place (d_out equal to d_in): the same numbers as from one
array into another, also where a row is computed in several overlapping blocks."""
import pytest

import paper_2101_05888_gb300 as sas

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(rows, n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn((rows, n, 2), device="cuda", generator=g))


@pytest.mark.parametrize("rows,n,L", [(300, 200, 50),        # one block a row
                                      (300, 2000, 1000),     # two
                                      (64, 5000, 200),       # several
                                      (700, 16384, 128),     # 92 MB: the copy is made in two runs of rows
                                      (1, 9000000, 64)])     # a row longer than a run
def test_matched_filter_in_place(rows, n, L):
    raw, rep = _rows(rows, n, 1), _rows(1, L, 2).reshape(-1)
    out = torch.empty_like(raw)
    sas.sas_matched_filter(raw, rows, n, rep, L, out)
    sas.sas_matched_filter(raw, rows, n, rep, L, raw)
    assert torch.equal(torch.view_as_real(out), torch.view_as_real(raw))


@pytest.mark.parametrize("rows,n", [(50, 64), (9001, 32)])
def test_whitening_and_gain_in_place(rows, n):
    e = _rows(rows, n, 3)
    a, b = torch.empty_like(e), e.clone()
    sas.sas_whiten(e, a, rows, n, 0.1)
    sas.sas_whiten(b, b, rows, n, 0.1)
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    sas.sas_tvg(a, e, rows, n, 0.5)
    sas.sas_tvg(b, b, rows, n, 0.5)
    assert torch.equal(torch.view_as_real(e), torch.view_as_real(b))
