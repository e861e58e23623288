"""The id-ordered subproblem kernels (k <= 6, out-degree up to 1024) against the
oracle: sizes at the edges of their words, tiles and size classes, every form
of the ring, and batches of mixed k.  Everything is exact."""
import numpy as np
import pytest

import oracle
from tests.graphs import gnp

pytestmark = pytest.mark.gpu
ORDS = ("color", "degree")


@pytest.fixture(scope="module")
def kcl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2203_13512_gb300 as kcl
    return kcl


# dense graphs: the first roots see almost all other vertices, so out-degrees
# and candidate sets run through every size up to about n * p
@pytest.mark.parametrize("n,p,ks", [
    (5, 0.9, (3, 4, 5)), (33, 0.9, (3, 4, 5, 6)), (36, 0.97, (3, 4, 5, 6)), (66, 0.8, (3, 4, 5, 6)),
    (67, 0.97, (4, 5)), (100, 0.7, (4, 5, 6)), (131, 0.95, (3, 4)), (133, 0.6, (5, 6)),
    (262, 0.5, (3, 4, 5)), (300, 0.9, (3, 4)), (530, 0.98, (3,)), (540, 0.3, (4, 5)), (1060, 0.96, (3,)),
])
def test_sizes(kcl, n, p, ks):
    rp, col = gnp(n, p, seed=n)
    g = kcl.kcl_load_csr(rp, col)
    for k in ks:
        ref = oracle.plain(rp, col, k)
        for o in ORDS:
            assert kcl.kcl_count(g, k, o) == ref[0], (k, o)
            assert kcl.kcl_list(g, k, o, None)[:2] == ref, (k, o)


def test_large_sets_match_the_list_form(kcl):
    """Candidate sets beyond a warp's shared matrix, k = 5 and 6, against the
    list form of SDegree (which these kernels do not run)."""
    rp, col = gnp(330, 0.8, seed=3)
    g, h = kcl.kcl_load_csr(rp, col), kcl.kcl_load_csr(rp, col)
    kcl.kcl_set_tuning(h, {"sdegree_bitmap": [0xFFFFFFFF] * kcl.KCL_MAX_CLASSES})
    for k in (4, 5):
        want = kcl.kcl_list(h, k, "degree", None)[:2]
        for o in ORDS:
            assert kcl.kcl_list(g, k, o, None)[:2] == want
            assert kcl.kcl_count(g, k, o) == want[0]
    want = kcl.kcl_count(h, 6, "degree")
    assert [kcl.kcl_count(g, 6, o) for o in ORDS] == [want, want]


@pytest.mark.parametrize("k", [3, 4, 5, 6])
@pytest.mark.parametrize("offset", [0, 1])
def test_ring_forms(kcl, k, offset):
    """Aligned and unaligned rings: exact room, truncated, wrapping with room
    for a part and for fewer records than a row of the matrix holds."""
    import torch
    rp, col = gnp(80, 0.6, seed=k)
    count, checksum = oracle.plain(rp, col, k)
    adj = np.zeros((80, 80), bool)
    for u in range(80):
        adj[u, col[rp[u]:rp[u + 1]]] = True
    g = kcl.kcl_load_csr(rp, col)

    def records(cap, wrap, order):
        buf = torch.zeros(cap * k + offset, dtype=torch.int32, device="cuda")[offset:]
        got = kcl.kcl_list(g, k, order, buf, wrap=wrap)
        rec = buf.cpu().numpy().reshape(-1, k)
        assert got[:2] == (count, checksum) and got[2] == min(count, cap) and got[3] == (cap < count and not wrap)
        if wrap:  # records that share a slot may be written at the same time
            return rec
        assert (np.diff(rec, axis=1) > 0).all()
        for i in range(k):
            for j in range(i):
                assert adj[rec[:, i], rec[:, j]].all()
        return rec

    for order in ORDS:
        assert len(np.unique(records(count, False, order), axis=0)) == count
        assert len(np.unique(records(count // 2, False, order), axis=0)) == count // 2
        records(count // 3, True, order)
        records(7, True, order)


def test_batch_of_mixed_k(kcl):
    rng = np.random.default_rng(4)
    members = [(gnp(int(n), float(p), seed=i), int(k)) for i, (n, p, k) in enumerate(
        zip(rng.integers(4, 160, 24), rng.uniform(0.2, 0.7, 24), rng.integers(3, 7, 24)))]
    gs = [kcl.kcl_load_csr(*m[0]) for m in members]
    ords = [ORDS[i % 2] for i in range(len(gs))]
    b = kcl.kcl_batch_create()
    counts, cks = kcl.kcl_count_batch(b, gs, [m[1] for m in members], ords, checksums=True)
    want = [oracle.plain(*m[0], m[1]) for m in members]
    assert list(zip(counts, cks)) == want
    assert kcl.kcl_count_batch(b, gs, [m[1] for m in members], ords)[0] == [w[0] for w in want]
