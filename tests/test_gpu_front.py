"""Pre-Core, Pre-List and the orientation, stage by stage against the oracle,
on graphs made for their rules: components that are cliques, that nearly are
(regular, or agreeing in degree and smallest id without being closed), rows
with long dead prefixes, rows beyond the kept 64 entries, and long Pre-Core
cascades."""
import numpy as np
import pytest

import kclgen
import oracle

pytestmark = pytest.mark.gpu


def _union(parts, seed):
    """Disjoint union of (n, edges), ids shuffled."""
    e, at = [], 0
    for n, edges in parts:
        if len(edges):
            e.append(np.asarray(edges, np.int64).reshape(-1, 2) + at)
        at += n
    perm = np.random.default_rng(seed).permutation(at) if seed else np.arange(at)
    return kclgen.from_edges(at, perm[np.concatenate(e)])


def _clique(n, drop=()):
    return n, [(u, v) for u in range(n) for v in range(u + 1, n) if (u, v) not in drop]


def _components():
    parts = [_clique(n) for n in (1, 2, 3, 4, 5, 6, 8, 16, 31, 32, 33, 34, 64, 65)]
    parts += [_clique(n, {(0, n - 1)}) for n in (4, 5, 33)] + [_clique(n, {(n - 2, n - 1)}) for n in (4, 6)]
    parts += [(n, [(i, (i + 1) % n) for i in range(n)]) for n in (4, 5, 50)]          # cycles
    parts += [(40, [(i, (i + d) % 40) for i in range(40) for d in (1, 2)])]            # 4-regular ring
    parts += [(8, [(u, v) for u in range(8) for v in range(u + 1, 8) if v != u + 4])]  # K_8 minus a matching
    # 0 sees 1, 2 with equal degrees and smallest id 0 everywhere, but 1-3, 2-4 leave its neighbourhood
    parts += [(5, [(0, 1), (0, 2), (1, 3), (2, 4), (3, 4)])]
    return parts


def _dead_prefix():
    """A hub whose row starts with 300 leaves, in a clique; one such per clique size."""
    e, at = [], 0
    for size, leaves in ((4, 3), (5, 40), (6, 300)):
        m = [at + leaves + i for i in range(size)]
        e += [(at + i, m[0]) for i in range(leaves)] + [(m[i], m[j]) for i in range(size) for j in range(i + 1, size)]
        at += leaves + size
    return at, e


GRAPHS = {
    "components": lambda: _union(_components(), 0),
    "components_shuffled": lambda: _union(_components() * 3, 5),
    "one_clique": lambda: _union([_clique(700)], 2),
    "dead_prefix": lambda: _union([_dead_prefix()], 0),
    # a path of triangles hanging on a clique: Pre-Core removes it one by one at k = 4
    "cascade": lambda: _union([(1030, _clique(30)[1] + [(i, i + d) for i in range(29, 1027) for d in (1, 2)])], 0),
    "long_rows": lambda: _union([(900, [(u, v) for u in range(9) for v in range(u + 1, 900)]), _clique(200, {(0, 1)})], 3),
    "skewed": lambda: kclgen.rmat20(seed=8, scale=15),
}


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("which", sorted(GRAPHS))
def test_stages(which, flags):
    import paper_2203_13512_gb300 as kcl
    rp, col = GRAPHS[which]()
    n = len(rp) - 1
    g = kcl.kcl_load_csr(rp, col)
    kcl.kcl_set_options(g, flags)  # 1: no Pre-Core
    ks = (3,) if which == "one_clique" else (3, 4, 6)  # the oracle lists every clique of a component
    for k in ks:
        core = np.ones(n, np.uint8) if flags else oracle.precore(rp, col, k)
        pl = oracle.prelist(rp, col, k, core)
        for mode, order in enumerate(("degree", "color")):
            st = kcl.kcl_stage_info(g, k, order)
            assert np.array_equal(st["alive_core"], core)
            assert np.array_equal(st["alive_final"], pl["alive"])
            assert st["prelist_count"] == pl["count"]
            od = oracle.outdegrees(rp, col, pl["alive"], mode)
            assert np.array_equal(st["outdeg"], od) and st["max_outdeg"] == od.max()
    for k in ks[:2]:
        if which != "one_clique":
            ref = oracle.plain(rp, col, k)
            for order in ("degree", "color"):
                assert kcl.kcl_list(g, k, order, None)[:2] == ref
                assert kcl.kcl_count(g, k, order) == ref[0]
