"""The ranked kernels (SDegree, BitCol), which run k > 6 and, when asked for, lists at any
k: work splitting, leaf forms, bit-rows and warps per root, in the classes above 128
out-neighbours as well.  Everything is exact."""
import numpy as np
import pytest

import kclgen
import oracle
from tests.graphs import elementary_symmetric, gnp, turan

pytestmark = pytest.mark.gpu
ORDS = ("color", "degree")
LISTS = 0xFFFFFFFF
K = 7
# by their largest out-degree; few 7-cliques for their size, which the oracle lists in
# a second or two
PARTS = {"d267": (260, 260, 2, 2, 1, 1, 1), "d605": (600, 600, 1, 1, 1, 1, 1)}
GRAPHS = {"d60": lambda: gnp(110, 0.6, seed=3), "d133": lambda: gnp(450, 0.35, seed=1),
          "d267": lambda: turan(PARTS["d267"]), "d605": lambda: turan(PARTS["d605"])}
_cache = {}


def _graph(name):
    """(CSR, count and checksum, per-root counts per ordering) of a graph, computed once."""
    if name not in _cache:
        rp, col = GRAPHS[name]()
        ref = oracle.plain(rp, col, K)
        if name in PARTS:
            assert ref[0] == elementary_symmetric(PARTS[name], K)
        per = {o: (oracle.sdegree if o == "degree" else oracle.bitcol)(
            rp, col, K, per_root=True, count_only=True)["per_root"] for o in ORDS}
        _cache[name] = (rp, col), ref, per
    return _cache[name]


def _check(kcl, name, tuning, orders=ORDS, widest=129):
    import torch
    (rp, col), ref, per = _graph(name)
    g = kcl.kcl_load_csr(rp, col)
    kcl.kcl_set_tuning(g, {f: [v] * kcl.KCL_MAX_CLASSES for f, v in tuning.items()})
    kcl.kcl_enable_timing(g, True)
    for o in orders:
        assert kcl.kcl_count(g, K, o) == ref[0], o
        if name != "d60":  # a CTA class did the work
            assert any(c["roots"] and c["hi"] >= widest for c in kcl.kcl_last_timing(g)[2])
        assert kcl.kcl_list(g, K, o, None)[:2] == ref, o
        pr = torch.zeros(len(rp) - 1, dtype=torch.int64, device="cuda")
        kcl.kcl_count_per_root(g, K, o, pr)
        assert np.array_equal(pr.cpu().numpy().astype(np.uint64), per[o]), o


@pytest.fixture(scope="module")
def kcl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2203_13512_gb300 as kcl
    return kcl


@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_work_splitting(kcl, name, split):
    _check(kcl, name, {"sdegree_split": split, "bitcol_split": split})


@pytest.mark.parametrize("warps", [1, 3])
@pytest.mark.parametrize("name", ["d133", "d267", "d605"])
def test_warps_per_root(kcl, name, warps):
    _check(kcl, name, {"sdegree_cta_warps": warps, "bitcol_cta_warps": warps})


@pytest.mark.parametrize("bitmap", [1, 64, LISTS])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_bit_rows_and_lists(kcl, name, bitmap):
    _check(kcl, name, {"sdegree_bitmap": bitmap}, orders=("degree",))


@pytest.mark.parametrize("gallop", [0, 4_000_000_000])
@pytest.mark.parametrize("name", ["d60", "d133", "d267"])
def test_leaf_forms_on_lists(kcl, name, gallop):
    _check(kcl, name, {"sdegree_bitmap": LISTS, "sdegree_gallop": gallop, "sdegree_gallop_list": gallop},
           orders=("degree",))


@pytest.mark.parametrize("gallop", [0, 4_000_000_000])
def test_leaf_forms_on_lists_at_small_k(kcl, gallop):
    tune = {"sdegree_bitmap": LISTS, "sdegree_gallop": gallop, "sdegree_gallop_list": gallop}
    for ks, (rp, col) in (((3, 4, 6), kclgen.chung_lu(10000, 50000, 2.5, groups=20, group_size=(12, 12), seed=1)),
                          ((4, 5), kclgen.chung_lu(3000, 12000, 2.3, groups=3, group_size=(260, 260), group_p=0.45,
                                                   seed=260))):
        g = kcl.kcl_load_csr(rp, col)
        kcl.kcl_set_tuning(g, {f: [v] * kcl.KCL_MAX_CLASSES for f, v in tune.items()})
        for k in ks:
            ref = oracle.plain(rp, col, k)
            assert kcl.kcl_count(g, k, "degree") == ref[0]
            assert kcl.kcl_list(g, k, "degree", None)[:2] == ref
