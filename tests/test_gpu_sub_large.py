"""The id-ordered kernels on out-degrees up to their largest, 1,024: one CTA per SM,
rows of 24 to 32 words, matrices in global scratch.  Near-complete graphs (one edge
missing) have a closed form."""
import math

import numpy as np
import pytest

import kclgen

pytestmark = pytest.mark.gpu


def _near_complete(n):
    u, v = np.triu_indices(n, 1)
    return kclgen.from_edges(n, np.stack([u, v], 1)[1:].astype(np.uint32))


@pytest.mark.parametrize("n,ks", [(730, (4, 5)), (801, (4, 5)), (1025, (4, 5))])
def test_counts(n, ks):
    import paper_2203_13512_gb300 as kcl
    g = kcl.kcl_load_csr(*_near_complete(n))
    kcl.kcl_enable_timing(g, True)
    for k in ks:
        for o in ("color", "degree"):
            assert kcl.kcl_count(g, k, o) == math.comb(n, k) - math.comb(n - 2, k - 2)
            assert max(c["hi"] for c in kcl.kcl_last_timing(g)[2] if c["roots"]) == n - 2


@pytest.mark.parametrize("n,k", [(730, 4), (1025, 4)])
def test_listings(n, k):
    """Checksums against SDegree's list form (other kernels)."""
    import paper_2203_13512_gb300 as kcl
    rp, col = _near_complete(n)
    g, h = kcl.kcl_load_csr(rp, col), kcl.kcl_load_csr(rp, col)
    kcl.kcl_set_tuning(h, {"sdegree_bitmap": [0xFFFFFFFF] * kcl.KCL_MAX_CLASSES})
    want = kcl.kcl_list(h, k, "degree", None)[:2]
    assert want[0] == math.comb(n, k) - math.comb(n - 2, k - 2)
    for o in ("color", "degree"):
        assert kcl.kcl_list(g, k, o, None)[:2] == want
