"""The profile records of the march hold only while none of its sources has
changed: the scheduler, the sweep and the root it solves."""
import os
import re
import shutil

import bench

CSRC = os.path.join(bench.ROOT, "paper_1502_07303_gb300", "csrc")


def test_every_source_of_the_march_counts(tmp_path, monkeypatch):
    here = bench.march_source_sha()
    dst = tmp_path / "paper_1502_07303_gb300" / "csrc"
    shutil.copytree(CSRC, dst, ignore=shutil.ignore_patterns("__pycache__"))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.march_source_sha() == here
    for name in bench.MARCH_SOURCES:
        old = (dst / name).read_bytes()
        (dst / name).write_bytes(old + b"\n")
        assert bench.march_source_sha() != here, name
        (dst / name).write_bytes(old)


def test_the_list_covers_what_the_march_includes():
    """Of the headers fmm_march.cu includes (and those they include) only the
    shared declarations are left out."""
    seen, todo = set(), ["fmm_march.cu"]
    while todo:
        name = todo.pop()
        seen.add(name)
        with open(os.path.join(CSRC, name)) as f:
            todo += [n for n in re.findall(r'#include "(fmm_[a-z0-9_]+\.(?:h|cuh))"', f.read()) if n not in seen]
    assert seen - {"fmm_internal.h"} == set(bench.MARCH_SOURCES)
