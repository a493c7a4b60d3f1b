"""The hash that ties committed profile figures to the kernel sources covers
every file the sweep units include, and moves with each of them."""
import os
import re
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_1206_0919_gb300", "csrc")


def included(name, seen):
    if name in seen:
        return
    seen.add(name)
    with open(os.path.join(CSRC, name)) as fh:
        for inc in re.findall(r'^\s*#include "([^"]+)"', fh.read(), re.M):
            if os.path.exists(os.path.join(CSRC, inc)):
                included(inc, seen)


def test_every_included_source_is_hashed(tmp_path, monkeypatch):
    units = [f for f in os.listdir(CSRC) if f.endswith(".cu") and f.startswith(("sweep", "tile"))]
    seen = set()
    for u in units:
        included(u, seen)
    assert {"sweep_f64.cu", "sweep_lines64.cuh", "fp64_math.cuh", "eos64.cuh", "eos_table.cuh", "chain.cuh",
            "sweep_tile.cuh", "tile_plan.h", "lines_plan.h"} <= seen
    assert seen <= {os.path.basename(f) for f in bench.kernel_sources()}

    copy = tmp_path / "paper_1206_0919_gb300" / "csrc"
    shutil.copytree(CSRC, copy)
    base = bench.kernel_source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_hash() == base
    hashes = {base}
    for f in sorted(seen):
        with open(copy / f, "a") as fh:
            fh.write("//\n")
        hashes.add(bench.kernel_source_hash())
    assert len(hashes) == len(seen) + 1
