"""The digest that recorded counters carry sees every file whose code the sweeps are compiled from,
and no comment."""
import os
import re
import shutil

import bench

CSRC = os.path.join("paper_1707_00198_gb300", "csrc")


def _included(name, seen):
    # project headers that a source file takes in, but for the interface of the host runtime
    text = open(os.path.join(bench.ROOT, CSRC, name), encoding="utf-8").read()
    for f in re.findall(r'#include "(\w+\.c?uh|\w+\.h)"', text):
        if f not in seen and os.path.exists(os.path.join(bench.ROOT, CSRC, f)):
            seen.add(f)
            _included(f, seen)
    return seen


def test_an_edit_of_the_sweeps_code_changes_the_digest(tmp_path, monkeypatch):
    files = {"lbcg_kernels.cu"} | {f for f in _included("lbcg_kernels.cu", set()) if f not in ("lbcg_internal.h", "lbcg_plan.h")}
    assert {"lbcg_device.cuh", "lbcg_node.cuh", "lbcg_geom.h"} <= files
    want = bench.kernel_source_digest()
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_digest() == want
    for f in sorted(files):
        path = tmp_path / CSRC / f
        text = path.read_text(encoding="utf-8")
        path.write_text("// a comment\n\n" + text + "\n  // another\n", encoding="utf-8")
        assert bench.kernel_source_digest() == want, f
        path.write_text(text + "\nint an_edit;\n", encoding="utf-8")
        assert bench.kernel_source_digest() != want, f
        path.write_text(text, encoding="utf-8")
