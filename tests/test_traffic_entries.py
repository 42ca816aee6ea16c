"""The DRAM traffic that bench.py reports with its lines was captured on the
kernels as they are: the entries of the committed table match the sources.
An ST entry depends on no FV-only header, so that FV work does not void it."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
import bench  # noqa: E402

with open(os.path.join(ROOT, "profiles", "traffic.json")) as fh:
    TABLE = {k: v for k, v in json.load(fh).items() if k != "_doc"}


@pytest.mark.parametrize("key", sorted(k for k in TABLE if "st" in k.split("|")[1].split("_")[0] or "rb3d" in k))
def test_streaming_and_3d_entries_are_current(key):
    e = TABLE[key]
    assert bench.measured_traffic(*key.split("|")) == e["bytes"]
    assert os.path.exists(os.path.join(ROOT, e["profile"]))


@pytest.mark.parametrize("key", sorted(k for k in TABLE if k.startswith("st ")))
def test_streaming_entries_hang_on_shared_headers_only(key):
    src = open(os.path.join(ROOT, "paper_1505_03271_gb300", "csrc", TABLE[key]["files"][0])).read()
    included = {line.split('"')[1] for line in src.splitlines() if line.startswith('#include "lb')}
    assert included == {"lb_pair.cuh"} and set(TABLE[key]["files"][1:]) == {"lb_pair.cuh", "lb_internal.cuh"}
    for h in ("lb_pair.cuh", "lb_internal.cuh"):
        text = open(os.path.join(ROOT, "paper_1505_03271_gb300", "csrc", h)).read()
        assert "launch_fv" not in text and "LaneMom" not in text
