"""Which layouts the binding takes (api._flat, api._rows), against the rule as it is
documented: any [kmax+1, n] view with unit column stride (any stride where n <= 1),
flattened inputs in row-major order."""
import pytest
import torch

from paper_2512_10059_gb300 import api


@pytest.mark.parametrize("kmax", [0, 1, 4])
@pytest.mark.parametrize("n", [0, 1, 2, 7])
def test_rows_accepts_unit_column_stride_only(kmax, n):
    rows = kmax + 1
    big = torch.zeros(rows + 2, 2 * n + 3)
    for out in (torch.empty(rows, n), big[:rows, :n], big[1:rows + 1, 1:n + 1], big[:rows, :2 * n:2],
                torch.empty(n, rows).t(), torch.empty(n).expand(rows, n), torch.empty(rows, n + 1),
                torch.empty(rows + 1, n), torch.empty(rows * n), torch.empty(rows, n, 1)):
        ok = out.dim() == 2 and out.shape[0] == rows and out.shape[1] == n and (n <= 1 or out.stride(1) == 1)
        if ok:
            assert api._rows(out, kmax, n) == (out.stride(0) if kmax > 0 else max(n, 1))
        else:
            with pytest.raises(ValueError):
                api._rows(out, kmax, n)


def test_flat_keeps_row_major_order():
    a = torch.arange(24.0)
    for t in (a, a[1:9], a[::2], a.view(4, 6), a.view(4, 6).t(), a.view(2, 3, 4)[:, 1], a[:0], a[5:6], a[3].view(())):
        f = api._flat(t)
        assert f.dim() == 1 and f.is_contiguous() and torch.equal(f, t.reshape(-1))
    assert api._flat(a) is a
