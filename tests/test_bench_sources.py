"""What bench.py's stored DRAM traffic is tied to (CPU only): the hash of a
kernel family covers every source its kernels are compiled from, and a capture
of either z pass is taken for the z pass."""

import csv
import json
import os
import re
import shutil

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_2606_01114_gb300", "csrc")


def closure(*names):
    """The sources and every header of csrc/ they include, directly or not."""
    seen, todo = set(), list(names)
    while todo:
        fn = todo.pop()
        if fn in seen:
            continue
        seen.add(fn)
        with open(os.path.join(CSRC, fn)) as f:
            todo += [h for h in re.findall(r'^#include "([^"]+)"', f.read(), re.M) if "/" not in h]
    return seen


@pytest.mark.parametrize("family,sources", [("demag", ("mm_demag.cu", "mm_zline.cu")), ("stage", ("mm_llg.cu",))])
def test_the_hash_covers_every_source_of_a_family(family, sources):
    assert closure(*sources) <= set(bench.KERNEL_SOURCES[family])


def test_the_register_z_pass_is_taken_for_the_z_pass(tmp_path, monkeypatch):
    dst = tmp_path / "paper_2606_01114_gb300" / "csrc"
    dst.mkdir(parents=True)
    for fn in set(sum(bench.KERNEL_SOURCES.values(), ())):
        shutil.copy(os.path.join(CSRC, fn), dst / fn)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    with open(tmp_path / "raw.csv", "w", newline="") as f:
        w = csv.writer(f)
        w.writerow(["Kernel Name", "dram__bytes_read.sum", "dram__bytes_write.sum"])
        w.writerow(["", "Mbyte", "Mbyte"])
        w.writerow(["void mm::k_zline<mm::ff, 8, 4, 0, 32, 256, 2>(mm::ffc *)", "400.0", "200.0"])
    assert bench.ingest_ncu(str(tmp_path / "raw.csv"), "ff", "film512 test") == 0
    t = json.load(open(tmp_path / "profiles" / "traffic.json"))
    assert t["zconv/ff"]["bytes_per_launch"] == 600 * 10 ** 6


def test_a_mode_does_not_report_the_plain_passes_traffic(monkeypatch):
    monkeypatch.setattr(bench, "source_hash", lambda k: "same")
    monkeypatch.setattr(bench.json, "load", lambda f: {"zconv/f32": {"bytes_per_launch": 1, "source_sha": "same"}})
    t = {m: bench.hbm_roofline("zconv", {"zconv": (1.0, 1)}, (512, 512, 16), 4, 1.0, "x", bench.traffic_key("f32", m))["traffic"]
         for m in ("fp32", "tf32", "bf16", "f4")}
    assert t == {"fp32": 1.0, "tf32": None, "bf16": None, "f4": None}
