"""CPU tests of the bench's candidate tables: every kind of plan that the planner returns is among the candidates, under
the name that plan_name gives it, and one-CTA plans of any kind count as plans without DSMEM."""
import os
import sys
import types

import pytest

from paper_2609_01864_gb300 import build as B
from paper_2609_01864_gb300 import credit as C

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.fixture()
def stub(monkeypatch):
    """The binding with every plan legal, a whole-row kernel at P <= 4, and no GPU asked."""
    B.build()
    import torch
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: types.SimpleNamespace(multi_processor_count=152))
    c = types.SimpleNamespace(**{k: getattr(C, k) for k in dir(C) if k.isupper()}, make_plan=C.make_plan)
    c.plan_check = lambda op, x, y, p, **kw: C.OK
    c.plan_kernel = lambda op, x, y, p, **kw: "k_row_team" if p.retain == C.RETAIN_ROW and p.cluster_size <= 4 else "k_ring"
    c.max_clusters = lambda *a, **kw: 8
    return c


def test_candidates_hold_the_planners_kinds_of_plans(stub):
    cands = bench.candidates(stub, C.SOFTMAX, None, None, fills=False)
    names = [n for n, _ in cands]
    assert len(set(names)) == len(names)
    assert {"one_cta_row", "cluster2_row", "cluster4_row", "one_cta_w8", "one_cta_w16", "cluster8_w8", "cluster8_w16",
            "cluster16_tm", "two_pass_g4"} <= set(names)
    assert "cluster8_row" not in names  # would run as the ring, which is there already
    assert [bench.plan_name(stub, p) for _, p in cands] == names


def test_rows_over_warps_without_threads_are_sixteen_warps(stub):
    assert bench.plan_name(stub, C.make_plan(C.PATH_CLUSTER, 8, retain=C.RETAIN_WARPS)) == "cluster8_w16"


def test_whole_rows_in_one_cta_are_no_dsmem_plans():
    r = bench.table_row("softmax", 4096, 1e9, {"one_cta_row": 1.0, "one_cta_w16": 1.5, "cluster4_row": 0.9, "two_pass_g1": 2.0},
                        1.0, "one_cta_row", 6800.0)
    assert r["best_non_dsmem_ms"] == 1.0 and r["speedup_vs_best_non_dsmem"] == 1.0 and r["best"] == "cluster4_row"


def test_tables_stay_off_the_result_line(capsys):
    import json
    tables = {"backward": {"shapes": [{"candidates": {f"c{i}": 0.1234 for i in range(30)}} for _ in range(28)]}}
    bench.emit({"metric": "m", "value": 1.0}, tables)
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": "m", "value": 1.0} and out.count("\n") == 1
    assert json.loads(err)["tables"] == tables
