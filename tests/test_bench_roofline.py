"""bench.py reports the dedispersion kernel that ran: the captured issue and
traffic figures are the shared-sum kernel's, the tile shape is the direct one's."""
import json
from types import SimpleNamespace

import bench
from paper_2606_27262_gb300 import build as spbuild


def test_fields_of_the_kernel_that_ran(tmp_path, monkeypatch):
    spbuild.build()
    prof = {"kernel_source_sha256_16": bench.kernel_source_hash(), "n_out": 4096,
            "dram_bytes_per_launch_full_config": 8e9, "lane_instructions_per_add": 0.4}
    path = tmp_path / "prof.json"
    path.write_text(json.dumps(prof))
    monkeypatch.setattr(bench, "PROFILE_JSON", str(path))
    plan = SimpleNamespace(shape=1, ntiles=7)
    direct = bench.ran_kernel(False, plan, 20.0, 152, 4096)
    assert direct["kernel"] == "dedisperse_kernel" and direct["traffic"] is None and direct["issue"] is None
    assert direct["kernel_shape"]["dm_tiles"] == 7 and direct["kernel_shape"]["shape"] == 1
    sums = bench.ran_kernel(True, plan, 60.0, 152, 4096)
    assert sums["kernel"] == "dedisp_sums_kernel" and sums["traffic"] == 8e9 and "kernel_shape" not in sums
    assert abs(sums["issue"]["achieved"] - 24.0) < 1e-9
    # another length, or sources that changed since the capture
    assert bench.ran_kernel(True, plan, 60.0, 152, 5000)["traffic"] is None
    path.write_text(json.dumps(prof | {"kernel_source_sha256_16": "0"}))
    stale = bench.ran_kernel(True, plan, 60.0, 152, 4096)
    assert stale["traffic"] is None and stale["issue"] is None
