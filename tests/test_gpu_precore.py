"""Pre-Core's rounds against the oracle where one batch of launches is not enough
(more wide rounds than that), and calls that run beside a long one on another
stream: no stage may wait for room that the long one does not leave."""
import threading
import time

import numpy as np
import pytest

import kclgen
import oracle
from tests.graphs import complete, disjoint_union, gnp

pytestmark = pytest.mark.gpu
ORDS = ("color", "degree")


def _unravelling(width, layers):
    """Layers of `width` vertices, each with two neighbours in the layer below and
    two in the one above: at k = 4 both end layers leave, then the next ones, one
    round of 2 * width vertices after another.  Beside them a dense random graph and
    a clique component (which Pre-List counts, once)."""
    i = np.arange(width * (layers - 1))
    up = i + width
    right = up - up % width + (up + 1) % width
    e = np.concatenate([np.stack([i, up], 1), np.stack([i, right], 1)])
    dense = disjoint_union(gnp(60, 0.7, seed=2), complete(7))
    n = width * layers
    src = np.repeat(np.arange(67), np.diff(dense[0].astype(np.int64)))
    pairs = np.stack([src, dense[1].astype(np.int64)], 1) + n
    return kclgen.from_edges(n + 67, np.concatenate([e, pairs[pairs[:, 0] < pairs[:, 1]]]))


# 2 * width below and above the width that a launch's last block takes on; rounds that
# fit the first launches, one more group of them and several
@pytest.mark.parametrize("width,layers", [(20, 11), (900, 40), (1500, 20), (1500, 60), (5000, 12)])
def test_many_wide_rounds(width, layers):
    import paper_2203_13512_gb300 as kcl
    rp, col = _unravelling(width, layers)
    g = kcl.kcl_load_csr(rp, col)
    want = oracle.plain(rp, col, 4)
    core = np.asarray(oracle.precore(rp, col, 4))
    for o in ORDS:
        st = kcl.kcl_stage_info(g, 4, o)
        assert np.array_equal(st["alive_core"], core) and st["prelist_count"] == 35
        assert kcl.kcl_count(g, 4, o) == want[0]
        assert kcl.kcl_list(g, 4, o, None)[:2] == want
    other = gnp(80, 0.3, seed=1)
    h = kcl.kcl_load_csr(*other)
    got = kcl.kcl_count_batch(kcl.kcl_batch_create(), [h, g], [3, 4], ["color"] * 2, checksums=True)
    assert list(zip(*got)) == [oracle.plain(*other, 3), want]


# the long call: k = 9 counts, whose kernels leave whole SMs idle, and a k = 7
# listing, whose kernels sit on every SM with half of its registers
@pytest.mark.parametrize("order,scale,long_call,k", [
    ("degree", 17, "kcl_count", 9), ("color", 17, "kcl_count", 9), ("color", 18, "kcl_list", 7)])
def test_calls_beside_a_long_one(order, scale, long_call, k):
    """A call of a few ms on one stream while another stream's kernels run for 4 s
    (R-MAT 18, cut by its time limit): it must not wait for their end."""
    import torch
    import paper_2203_13512_gb300 as kcl
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        long_g = kcl.kcl_load_csr(*kclgen.rmat20(seed=1, scale=18))
    with torch.cuda.stream(b):
        g = kcl.kcl_load_csr(*kclgen.rmat20(seed=3, scale=scale))
    want = kcl.kcl_count(g, 5, order)

    def run_long():
        if long_call == "kcl_list":
            kcl.kcl_list(long_g, k, "color", None)
        else:
            kcl.kcl_count(long_g, k, "degree")

    kcl.kcl_set_time_limit(long_g, 1)  # loads the kernels, which waits for running ones
    with pytest.raises(kcl.KclError):
        run_long()
    kcl.kcl_set_time_limit(long_g, 4000)
    status = []

    def run():
        try:
            run_long()
        except kcl.KclError as e:
            status.append(e.status)

    t = threading.Thread(target=run)
    t.start()
    time.sleep(0.3)
    start = time.perf_counter()
    got = kcl.kcl_count(g, 5, order)
    took = time.perf_counter() - start
    alive = t.is_alive()
    t.join()
    assert got == want and status == [kcl.KCL_ETIMEOUT]
    assert alive and took < 2.0
