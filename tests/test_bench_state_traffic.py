"""Host logic of bench.py: the state kernel's ncu traffic figure is used only
for the kernel source it was taken on."""
import json
import os

import bench


def test_state_traffic_figure_only_for_its_kernel_source(monkeypatch):
    with open(os.path.join(bench.ROOT, "profiles", "k_state_print_traffic.json")) as f:
        d = json.load(f)
    monkeypatch.setattr(bench, "_state_source_sha", lambda: d["kernel_sha"])
    assert bench._state_traffic_per_site() == d["dram_bytes_per_site"]
    monkeypatch.setattr(bench, "_state_source_sha", lambda: "0000000000000000")
    assert bench._state_traffic_per_site() is None
