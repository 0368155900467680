"""What the autotuner keeps belongs to the kernels it was measured on: entries of other sources (or
without a mark of theirs) are not used."""
import json

from paper_1104_5497_gb300 import autotune as A


def test_entries_of_other_kernels_are_not_found(tmp_path, monkeypatch):
    path = str(tmp_path / "autotune.json")
    with open(path, "w") as fh:
        json.dump({"N=10|GPU X|sms=152": dict(blocks_per_sm=7, list_blocks_per_sm=2)}, fh)
    assert A.load_cache(path).get(A.cache_key(10, "GPU X", 152)) is None
    A.store_cache(path, A.cache_key(10, "GPU X", 152), dict(blocks_per_sm=8, list_blocks_per_sm=2))
    assert A.load_cache(path)[A.cache_key(10, "GPU X", 152)]["blocks_per_sm"] == 8
    mine = A.cache_key(10, "GPU X", 152)
    monkeypatch.setattr(A, "kernels", lambda: "0123456789abcdef")
    assert A.cache_key(10, "GPU X", 152) != mine
    assert A.load_cache(path).get(A.cache_key(10, "GPU X", 152)) is None


def test_the_mark_follows_the_sources(tmp_path, monkeypatch):
    pkg = tmp_path / "pkg"
    (pkg / "csrc").mkdir(parents=True)
    for f in ("xy_track.cuh", "nphc_api.cu", "quad.cuh"):
        (pkg / "csrc" / f).write_text("a")
    monkeypatch.setattr(A, "__file__", str(pkg / "autotune.py"))
    read = A.kernels.__wrapped__
    first = read()
    (pkg / "csrc" / "quad.cuh").write_text("b")       # no tracker of the ring's
    assert read() == first
    (pkg / "csrc" / "xy_track.cuh").write_text("b")
    assert read() != first


def test_four_lane_candidates_are_whole_blocks():
    assert {12, 8, 4} <= set(A.FP32_CANDIDATES) and A.FP32_CANDIDATES[0] == 0
