"""The benchmark's DRAM figure is that of the kernel and the radii it timed,
and no autotuner candidate runs another one's kernel with the same radii."""
import json
import os

import bench

ROOT = os.path.dirname(os.path.abspath(bench.__file__))


def _record(tmp_path, monkeypatch, **changes):
    rec = json.load(open(bench.TRAFFIC_RECORD))
    rec = dict(rec, sources=bench.source_hashes(rec["sources"].keys()), **changes)
    p = tmp_path / "record.json"
    p.write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "TRAFFIC_RECORD", str(p))
    return rec


def test_traffic_only_of_the_captured_tuning(tmp_path, monkeypatch):
    rec = _record(tmp_path, monkeypatch, tuning=[8, 2, 0])
    assert bench.knn_traffic_per_particle((8, 2, 0)) == (rec["traffic_bytes_per_particle"], rec["basis"])
    # cells per radius do not reach the grouped kernel
    assert bench.knn_traffic_per_particle((8, 1, 0))[0] == rec["traffic_bytes_per_particle"]
    for other in ((4, 2, 0), (16, 2, 0), (8, 2, 3), (32, 2, 0)):
        value, why = bench.knn_traffic_per_particle(other)
        assert value is None and "tuning" in why


def test_the_record_names_its_tuning_and_the_boxes():
    rec = json.load(open(bench.TRAFFIC_RECORD))
    assert f"--qpw {rec['tuning'][0]} " in rec["capture"] and "lower bound" in rec["basis"]
    for name in ("knn_gq.cu", "boxtree.cu"):
        assert f"paper_1001_3411_gb300/csrc/{name}" in rec["sources"]


def test_candidates_differ():
    for name, cands in bench.CANDS.items():
        cases = [bench.knn_case(c) for c in cands]
        if name == "plain":      # one radius for every chunk
            cases = ["grouped" if c[0] in (4, 8, 16) and not c[2] else c for c in cases]
        assert len(set(cases)) == len(cases), name
