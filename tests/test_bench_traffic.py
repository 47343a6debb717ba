"""The DRAM traffic that the benchmark reports as measured is tied to every file
of the hopping kernels, not only to two of them.  No GPU."""
import json
import os
import re
import shutil

import bench

CSRC = os.path.join(bench.ROOT, "paper_2103_05034_gb300", "csrc")
HOST_ONLY = {"dwf_internal.cuh", "per_device.cuh", "dwfmg.h"}  # included by the kernels' files, no kernel text


def _closure(name, seen):
    if name in seen or name in HOST_ONLY:
        return seen
    seen.add(name)
    for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(os.path.join(CSRC, name)).read(), flags=re.M):
        _closure(os.path.basename(inc), seen)
    return seen


def test_the_hash_covers_what_the_hopping_kernels_include():
    used = set()
    for unit in ("dhop_f32.cu", "dhop_f16.cu", "dhop_f64.cu"):
        used |= _closure(unit, set()) - {unit}
    assert used - {"dfloat.cuh"} == {os.path.basename(f) for f in bench.HOP_KERNEL_SOURCES}


def test_a_change_of_any_kernel_file_drops_the_figure(tmp_path, monkeypatch):
    files = bench.HOP_KERNEL_SOURCES + ("profiles/traffic.json",)
    for f in files:
        os.makedirs(tmp_path / os.path.dirname(f), exist_ok=True)
        shutil.copy(os.path.join(bench.ROOT, f), tmp_path / f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    shash = bench.source_hash(*bench.HOP_KERNEL_SOURCES[1:3])  # the kernels' common file and the pair kernel's
    key, rec = next(iter(json.load(open(tmp_path / "profiles" / "traffic.json")).items()))
    assert bench.profile_traffic(key, shash) == rec["dram_bytes_per_launch"]
    for f in bench.HOP_KERNEL_SOURCES:
        text = open(tmp_path / f).read()
        (tmp_path / f).write_text(text + "// changed\n")
        assert bench.profile_traffic(key, shash) is None
        assert bench.profile_traffic(key, bench.source_hash(*bench.HOP_KERNEL_SOURCES[1:3])) is None
        (tmp_path / f).write_text(text)
