"""What the benchmark says about the round kernels: which sources its traffic record
belongs to, the cluster kernel's name, and which byte counts are rates."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1812_10499_gb300", "csrc")
HEADERS = sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh")) + ["sssp_engine.h"]


@pytest.fixture
def bench(monkeypatch):
    monkeypatch.syspath_prepend(ROOT)
    import bench
    return bench


@pytest.mark.parametrize("header", HEADERS)
def test_hash_follows_every_kernel_header(bench, tmp_path, monkeypatch, header):
    dst = tmp_path / "paper_1812_10499_gb300" / "csrc"
    shutil.copytree(CSRC, dst)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_source_sha256()
    with open(dst / header, "a") as f:
        f.write("\nint one_more;\n")
    assert bench.kernel_source_sha256() != before


def test_cluster_kernel_by_rule(bench):
    small = {r for r in bench.RULES if bench.tail_kernel(r) == "k_small"}
    assert small == {"thr", "mind", "thr-cheap", "mind-cheap", "thr-win", "mind-win", "thr-cheap-win"}
    assert all(bench.tail_kernel(r) == "k_tail" for r in set(bench.RULES) - small)


def test_whole_row_counts_are_no_rate(bench):
    """The lower-bound kernel reads less than its counters say: no fraction of the peak."""
    ctr = {"out_scanned": 1000, "front_visits": 10, "in_scanned": 5000, "active_visits": 20}
    prof = {"grid_counters": ctr, "tail_counters": ctr, "cupdate_ms": 2.0, "cupdate_launches": 4,
            "relax_ms": 1.0, "relax_launches": 4, "tail_ms": 1.0, "tail_launches": 4}
    t = bench.kernel_table(prof, "thr-cheap", 1000.0)
    assert set(t) == {"k_cupdate", "k_relax", "k_small"}
    assert "frac" not in t["k_cupdate"] and "achieved_gbs" not in t["k_cupdate"]
    assert t["k_cupdate"]["equivalent_gbs"] == pytest.approx((24 * 5000 + 48 * 20) / 2e-3 / 1e9)
    assert t["k_relax"]["frac"] == pytest.approx((16 * 1000 + 36 * 10) / 1e-3 / 1e9 / 1000.0)
    assert [t[k]["share"] for k in ("k_cupdate", "k_relax", "k_small")] == [0.5, 0.25, 0.25]
