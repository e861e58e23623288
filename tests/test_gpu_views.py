"""Calls on a graph view whose workspace does not exist yet."""
import numpy as np
import pytest

import oracle
from tests.graphs import gnp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["color", "degree"])
def test_count_roots_is_a_views_first_call(order):
    import torch
    import paper_2203_13512_gb300 as kcl
    rp, col = gnp(70, 0.5, seed=3)
    g = kcl.kcl_load_csr(rp, col)
    roots = np.arange(0, 70, 3, dtype=np.uint32)
    mode = oracle.bitcol if order == "color" else oracle.sdegree
    want = mode(rp, col, 4, roots=roots, per_root=True, count_only=True)["per_root"]
    view = kcl.kcl_graph_view(g)
    for h in (view, g, view):
        per = torch.zeros(70, dtype=torch.int64, device="cuda")
        total = kcl.kcl_count_roots(h, 4, order, roots, per)
        assert np.array_equal(per.cpu().numpy().astype(np.uint64), want) and total == int(want.sum())
