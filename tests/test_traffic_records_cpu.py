"""The recorded DRAM traffic of a kernel is void once any file that its device
code is in has changed: the key covers the kernel's file and every .cuh that
it reaches through includes."""
import json
import os
import re

import pytest

from paper_0902_3185_gb300 import prof

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0902_3185_gb300", "csrc")


def reached(f):
    txt = open(os.path.join(CSRC, f)).read()
    out = {f}
    for inc in re.findall(r'#include "([^"]+\.cuh)"', txt):
        out |= reached(inc)
    return out


@pytest.mark.parametrize("name", sorted(prof.TRAFFIC_KERNELS))
def test_key_covers_every_device_source(name):
    got = {os.path.basename(f) for f in prof.traffic_sources(name)}
    assert reached(prof.TRAFFIC_KERNELS[name]) <= got


def test_the_shared_tile_is_part_of_both_cuda_core_products():
    for name in ("fp64_product", "df64_product_real"):
        assert any(f.endswith("seg_tile.cuh") for f in prof.traffic_sources(name))


def test_a_record_lives_only_with_its_sources(tmp_path, monkeypatch):
    import bench
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    name = "df64_product_real"
    for f in prof.traffic_sources(name):
        os.makedirs(os.path.dirname(tmp_path / f), exist_ok=True)
        (tmp_path / f).write_bytes(open(os.path.join(ROOT, f), "rb").read())
    rec = {"dram_bytes_per_product": 7.0, "sources": [prof.traffic_sources(name)[0]],
           "source_sha": bench.source_sha(prof.traffic_sources(name))}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps({name: rec}))
    assert bench.recorded_traffic(name) == 7.0
    for f in prof.traffic_sources(name):
        was = (tmp_path / f).read_bytes()
        (tmp_path / f).write_bytes(was + b"\n// changed\n")
        assert bench.recorded_traffic(name) is None, f
        (tmp_path / f).write_bytes(was)
    assert bench.recorded_traffic("no such record") is None
