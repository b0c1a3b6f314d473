"""The reference arm of bench.py runs on the host alone and prints the contract's JSON line
(CPU only: the reference arm times the FP64 oracle, no GPU is involved)."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_json_line():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "small",
                        "--steps", "1", "--warmup", "1"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [l for l in r.stdout.splitlines() if l.strip().startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    for k in ("impl", "metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert k in d, k
    assert d["impl"] == "reference" and d["value"] > 0 and d["higher_is_better"] is True
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0


def test_profile_values_hold_for_their_rows_and_sources_only(tmp_path, monkeypatch):
    # a count taken on some rows and kernel sources is not applied to others: null instead
    import hashlib
    import bench
    src = tmp_path / "paper_2105_13611_gb300" / "csrc"
    src.mkdir(parents=True)
    (src / "k.cu").write_text("kernel")
    (tmp_path / "profiles").mkdir()
    sha = hashlib.sha1(b"kernel").hexdigest()
    (tmp_path / "profiles" / "p.md").write_text(f"rows: 3,5\nper: 0.25\nk_source_sha1: {sha}\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profile_value("p.md", "per", "k", ["k.cu"], [3, 5]) == 0.25
    assert bench.profile_value("p.md", "per", "k", ["k.cu"], [3, 6]) is None
    assert bench.profile_value("p.md", "per", "k", ["k.cu"], [3]) is None
    assert bench.profile_value("q.md", "per", "k", ["k.cu"], [3, 5]) is None
    (src / "k.cu").write_text("changed")
    assert bench.profile_value("p.md", "per", "k", ["k.cu"], [3, 5]) is None
