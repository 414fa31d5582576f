"""The kernel that bench.py names for a run without tuning is the one that the
choice it sets selects: every occurrence's row, one group of 32 events per
batch (FP64: two), whatever the row."""
import pytest

import bench


@pytest.mark.parametrize("prec,rows,want", [(1, (64, True), "k_rows_packed<16,1,1,fixed>"),
                                            (2, (64, False), "k_rows<16,1,2,fixed>"),
                                            (1, (32, True), "k_rows_packed<8,1,1,fixed>"),
                                            (0, (64, True), "k_rows64<8,2,fixed>")])
def test_the_record_of_an_untuned_run(monkeypatch, prec, rows, want):
    monkeypatch.setattr(bench, "hbm_peak", lambda: (6700.0, "measured"))
    monkeypatch.setattr(bench, "ncu_traffic", lambda key: None)
    r = bench.roofline(10**9, 10**6, 16, prec, 4.0, None, (2.9e11, [(1, 4, 3, 2.9e11)]), rows)
    assert r["kernel"] == want
