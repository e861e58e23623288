"""The degeneracy peel's rounds against the oracle where its rules change: one
CTA, one cluster, grid and cluster, thresholds past the near list's window and
gaps wider than it, rows longer than 4,096 in wide rounds, and more of those
than a round's list holds.  Both entry points."""
import numpy as np
import pytest

import kclgen
import oracle

pytestmark = pytest.mark.gpu


def _layers(hubs, links, ring):
    """30,000 first-layer vertices of degree links + 2 leave in round 0, the
    30,000 of the second layer (ring neighbours and two of the first) and the
    hubs, whose rows hold 30,000 links / hubs entries, together in round 1."""
    m = 30000
    i = np.arange(m)
    first, second = hubs + i, hubs + m + i
    e = [np.stack([first, second], 1), np.stack([first, np.roll(second, 1)], 1)]
    e += [np.stack([first, (i * links + z) % hubs], 1) for z in range(links)]
    e += [np.stack([second, np.roll(second, z + 1)], 1) for z in range(ring // 2)]
    return kclgen.from_edges(hubs + 2 * m, np.concatenate(e))


def _cliques(*sizes):
    """Near-cliques (no Pre-List shortcut) of the given sizes and a long cycle."""
    e, at = [], 0
    for s in sizes:
        u, v = np.triu_indices(s, 1)
        e.append(np.stack([at + u, at + v], 1)[1:])
        at += s
    i = np.arange(500)
    e.append(np.stack([at + i, at + (i + 1) % 500], 1))
    return kclgen.from_edges(at + 500, np.concatenate(e))


GRAPHS = {
    "cluster": lambda: kclgen.rmat20(seed=5, scale=18),
    "grid_and_cluster": lambda: kclgen.rmat20(seed=6, scale=19),
    "one_cta": lambda: kclgen.chung_lu(3000, 12000, 2.3, groups=5, group_size=(10, 40), seed=4),
    "gaps": lambda: _cliques(20, 53, 55, 150, 400),
    "long_rows": lambda: _layers(5, 1, 2),
    "many_long_rows": lambda: _layers(300, 41, 42),
}


@pytest.mark.parametrize("which", sorted(GRAPHS))
def test_rounds(which):
    import torch
    import paper_2203_13512_gb300 as kcl
    rp, col = GRAPHS[which]()
    n = len(rp) - 1
    g = kcl.kcl_load_csr(rp, col)
    st = kcl.kcl_stage_info(g, 3, "color")
    alive = st["alive_final"]
    want, _ = oracle.degeneracy_rounds(rp, col, alive)
    assert np.array_equal(st["key"], want)
    src = np.repeat(np.arange(n), np.diff(rp.astype(np.int64)))
    deg = np.bincount(src[(alive[src] == 1) & (alive[col] == 1)], minlength=n).astype(np.int32)
    out = torch.full((n,), 7, dtype=torch.int32, device="cuda")
    kcl.kcl_degeneracy_order_noalloc(
        torch.from_numpy(rp.astype(np.int64)).cuda(), torch.from_numpy(col.astype(np.int32)).cuda(),
        torch.from_numpy(alive).cuda(), torch.from_numpy(deg).cuda(), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
