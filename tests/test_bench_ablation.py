"""bench.py --form ablation, driven on the CPU with a stand-in for the library: which
calls each row makes."""
import argparse
import sys
import types

import torch

import bench
import kclgen
import paper_2203_13512_gb300 as real


class Graph:
    def __init__(self):
        self.flags, self.tune = 0, {}

    def free(self):
        pass


def test_the_prune_is_compared_where_its_kernels_run(monkeypatch):
    """Switching the colour prune off changes the kernels of k <= 6 altogether, so
    both sides of that row have to be calls with k > 6."""
    calls = []

    def count(g, k, order):
        calls.append((k, order, g.flags, tuple(sorted(g.tune))))
        return 7

    fake = types.SimpleNamespace(
        KCL_MAX_CLASSES=real.KCL_MAX_CLASSES, KCL_OPT_NO_PRECORE=real.KCL_OPT_NO_PRECORE,
        KCL_OPT_NO_PRELIST=real.KCL_OPT_NO_PRELIST, KCL_OPT_NO_COLOR_PRUNE=real.KCL_OPT_NO_COLOR_PRUNE,
        kcl_load_csr=lambda rp, col: Graph(), kcl_graph_view=lambda g: Graph(), kcl_count=count,
        kcl_enable_timing=lambda g, on: None, kcl_set_options=lambda g, f: setattr(g, "flags", f),
        kcl_set_tuning=lambda g, t: setattr(g, "tune", t), kcl_scratch_bytes=lambda g: (1, 2),
        kcl_last_timing=lambda g: ({"listing": 1.0, "total": 2.0}, {}, []))
    monkeypatch.setitem(sys.modules, "paper_2203_13512_gb300", fake)
    monkeypatch.setattr(bench, "workload", lambda: (None, None))
    monkeypatch.setattr(kclgen, "rmat20", lambda **kw: (None, None))
    monkeypatch.setattr(torch.cuda, "synchronize", lambda: None)
    out = bench.run_ablation(argparse.Namespace(steps=1))
    pruned = [c for c in calls if c[2] & real.KCL_OPT_NO_COLOR_PRUNE]
    assert pruned and all(k > 6 and order == "color" for k, order, _, _ in pruned)
    row, = [r for r in out["calls"].values() if "no colour prune" in r]
    assert {(k, order, 0, ()) for k, order, _, _ in pruned} <= set(calls)
    assert set(row) == {"all on", "no colour prune"}
    assert row["all on"] == {"listing": 1.0, "total": 2.0, "count": 7}
    for k in (4, 5):
        for o in ("color", "degree"):
            assert set(out["calls"]["k=%d %s" % (k, o)]) == {
                "all on", "no Pre-Core", "no Pre-List", "one warp per root (NodeParallel)"}
            assert out["scratch_bytes"]["k=%d %s" % (k, o)] == {"workspace": 1, "arena": 2}
