"""The degeneracy peel's rounds against the oracle by size of the graph: the cluster
alone, a grid that hands over at once (few vertices, many entries), and a grid that
walks rows longer than 4,096 entries itself."""
import numpy as np
import pytest

import kclgen
import oracle

pytestmark = pytest.mark.gpu


def _layers(m, hubs, links):
    """m first-layer vertices of degree links + 2 leave in round 0, the m of the second
    layer (two neighbours in it, two in the first) and the hubs, whose rows hold
    m * links / hubs entries, together in round 1."""
    i = np.arange(m)
    first, second = hubs + i, hubs + m + i
    e = [np.stack([first, second], 1), np.stack([first, np.roll(second, 1)], 1), np.stack([second, np.roll(second, 1)], 1)]
    e += [np.stack([first, (i * links + z) % hubs], 1) for z in range(links)]
    return kclgen.from_edges(hubs + 2 * m, np.concatenate(e))


def _dense(n, edges):
    rng = np.random.default_rng(n)
    e = rng.integers(0, n, (edges, 2))
    e[: edges // 4] //= 8  # a denser part, so that there are many thresholds
    e = np.sort(e[e[:, 0] != e[:, 1]], axis=1)
    key = np.unique(e[:, 0] * n + e[:, 1])
    return kclgen.from_edges(n, np.stack([key // n, key % n], 1))


GRAPHS = {
    "cluster": lambda: kclgen.rmat20(seed=5, scale=16),
    "dense": lambda: _dense(40_000, 2_300_000),
    "grid_long_rows": lambda: _layers(140_000, 5, 1),
    "grid_many_long_rows": lambda: _layers(140_000, 300, 10),
}


@pytest.mark.parametrize("which", sorted(GRAPHS))
def test_rounds(which):
    import torch
    import paper_2203_13512_gb300 as kcl
    rp, col = GRAPHS[which]()
    n = len(rp) - 1
    if which.startswith("grid"):  # both entry points leave round 1 to the grid
        assert np.diff(rp.astype(np.int64)).max() > 4096
    want, _ = oracle.degeneracy_rounds(rp, col)
    g = kcl.kcl_load_csr(rp, col)
    kcl.kcl_set_options(g, kcl.KCL_OPT_NO_PRECORE | kcl.KCL_OPT_NO_PRELIST)
    assert np.array_equal(kcl.kcl_stage_info(g, 3, "color")["key"], want)
    row = torch.from_numpy(rp.astype(np.int64)).cuda()
    out = torch.full((n,), 7, dtype=torch.int32, device="cuda")
    kcl.kcl_degeneracy_order_noalloc(row, torch.from_numpy(col.astype(np.int32)).cuda(),
                                     torch.ones(n, dtype=torch.uint8, device="cuda"),
                                     (row[1:] - row[:-1]).to(torch.int32), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
