"""The committed DRAM traffic record is reported only for the launches it was taken on: stacked steps, by the sources of
the kernel and of the rules that choose it."""
import json

import bench


def test_record_holds_for_stacked_steps_of_the_recorded_sources(tmp_path, monkeypatch):
    rec = {"sources_sha256": bench.traffic_digest(), "traffic_bytes_per_layer": {"4": 1000}}
    (tmp_path / "profiles").mkdir()
    for name in bench.TRAFFIC_SOURCES:
        (tmp_path / "paper_2609_03430_gb300" / "csrc").mkdir(parents=True, exist_ok=True)
        src = f"{bench.ROOT}/paper_2609_03430_gb300/csrc/{name}"
        (tmp_path / "paper_2609_03430_gb300" / "csrc" / name).write_bytes(open(src, "rb").read())
    (tmp_path / "profiles" / "attn_kernel_traffic.json").write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profiled_traffic(4, 64, "step") == 64000
    assert bench.profiled_traffic(4, 64, "layer") is None
    assert bench.profiled_traffic(3, 64, "step") is None
    with open(tmp_path / "paper_2609_03430_gb300" / "csrc" / "ra_api.cu", "a") as f:
        f.write("// another rule\n")
    assert bench.profiled_traffic(4, 64, "step") is None
