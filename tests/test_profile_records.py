"""The committed counter records belong to the sources they name: a record whose
source hash was replaced without a capture, or whose counters were, is not used."""
import glob
import hashlib
import json
import os

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _records():
    for path in sorted(glob.glob(os.path.join(ROOT, "profiles", "*.md"))):
        text = open(path).read()
        if "```json" in text:
            yield json.loads(text.split("```json", 1)[1].split("```", 1)[0])


def test_committed_records_are_as_captured():
    records = list(_records())
    assert {r["kernel"] for r in records} >= {"gather", "table"}
    for rec in records:
        assert rec.get("sha256") == bench.record_digest(rec), rec["kernel"]


def test_hash_or_counters_alone_void_a_record(tmp_path, monkeypatch):
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles").mkdir()
    (tmp_path / "k.cu").write_text("new source")
    now = hashlib.sha256(b"new source").hexdigest()

    def used(rec):
        (tmp_path / "profiles" / "r.md").write_text("# r\n```json\n" + json.dumps(rec) + "\n```\n")
        return bench.recorded_profile("gather") is not None

    rec = {"kernel": "gather", "source_files": ["k.cu"], "source_sha256": hashlib.sha256(b"old").hexdigest(),
           "traffic_bytes_per_launch": 5, "alu_warp_inst_per_unit": 2.5}
    assert not used(dict(rec, source_sha256=now))          # no digest: an older record with the hash replaced
    rec["sha256"] = bench.record_digest(rec)
    assert not used(rec)                                    # another source
    assert not used(dict(rec, source_sha256=now))           # the hash replaced alone
    rec["source_sha256"] = now
    rec["sha256"] = bench.record_digest(rec)
    assert used(rec)
    assert not used(dict(rec, traffic_bytes_per_launch=6))  # a counter replaced alone
