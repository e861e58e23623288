"""kcl_scratch_bytes counts every byte of device scratch once."""
import pytest

import kclgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["color", "degree"])
def test_the_small_arena_is_part_of_the_workspace(order):
    """A small graph's call allocates nothing beyond what loading did."""
    import paper_2203_13512_gb300 as kcl
    g = kcl.kcl_load_csr(*kclgen.chung_lu(2000, 9000, 2.3, groups=4, group_size=(10, 14), seed=7))
    loaded = kcl.kcl_scratch_bytes(g)
    assert loaded[1] == 0
    kcl.kcl_count(g, 4, order)
    called = kcl.kcl_scratch_bytes(g)
    assert called[1] > 0 and sum(called) == loaded[0]
