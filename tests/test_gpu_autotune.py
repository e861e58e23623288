"""The autotuner on calls of the id-ordered kernels (k <= 6): values that those kernels
do not use stay what they were; k > 6 tunes them all."""
import pytest

import kclgen
import oracle

pytestmark = pytest.mark.gpu
LISTS = 0xFFFFFFFF


def test_unused_values_are_kept():
    import paper_2203_13512_gb300 as kcl
    rp, col = kclgen.chung_lu(10000, 50000, 2.5, groups=20, group_size=(12, 12), seed=1)
    n = kcl.KCL_MAX_CLASSES
    own = {"sdegree_gallop": [77] * n, "sdegree_gallop_list": [78] * n, "sdegree_bitmap": [5] * n,
           "sdegree_split": [9] * n, "bitcol_split": [11] * n}
    g = kcl.kcl_load_csr(rp, col)
    for k, order, listing in ((5, "degree", False), (4, "degree", True), (6, "color", False), (3, "color", True)):
        kcl.kcl_set_tuning(g, own)
        t = kcl.kcl_autotune(g, k, order, listing)
        assert t == kcl.kcl_get_tuning(g)
        for c in range(n):
            assert t["sdegree_bitmap"][c] in (5, LISTS)
            if t["sdegree_bitmap"][c] == 5:  # id-ordered kernels
                assert [t[f][c] for f in ("sdegree_gallop", "sdegree_gallop_list", "sdegree_split")] == [77, 78, 9]
            assert t["bitcol_split"][c] == 11
    # lists set by hand: the other form is tried
    kcl.kcl_set_tuning(g, {"sdegree_bitmap": [LISTS] * n})
    t = kcl.kcl_autotune(g, 5, "degree")
    assert set(t["sdegree_bitmap"]) <= {0, LISTS}
    assert kcl.kcl_count(g, 5, "degree") == oracle.plain(rp, col, 5)[0]
    # k > 6: every candidate is tried, so the preset values are gone where there are roots
    kcl.kcl_set_tuning(g, own)
    t = kcl.kcl_autotune(g, 8, "degree")
    assert t["sdegree_gallop"][0] in (0, 40, 80, 160, 400) and t["sdegree_split"][0] in (0, 2, 8, 32)
