"""The binding addresses the rows of a (3, n) tensor from its base and stride:
the same addresses as the three indexed views, for every form it is given."""
import pytest
import torch

import paper_2206_02937_gb300 as cg


@pytest.mark.parametrize("form", ["plain", "columns", "transposed", "more_rows", "float64", "list", "flat"])
def test_rows_match_indexed_views(form):
    base = torch.zeros(3, 40)
    t = {"plain": base, "columns": base[:, 7:23], "transposed": torch.zeros(40, 3).T, "more_rows": torch.zeros(5, 9),
         "float64": base.double(), "list": [torch.zeros(4), torch.zeros(4), torch.zeros(4)],
         "flat": torch.zeros(3)}[form]
    assert cg._rows(t) == tuple(t[i].data_ptr() for i in range(3))


def test_two_rows_are_refused():
    with pytest.raises(IndexError):
        cg._rows(torch.zeros(2, 40))
    assert cg._ptr(None) == 0
