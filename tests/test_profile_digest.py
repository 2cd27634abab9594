"""The digest that ties the plane pass's captured traffic to its sources covers every device header the
kernel is made of (CPU only): a step changed in any of them makes the captured figure stale."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1406_7803_gb300", "csrc")


def included(name, seen):
    if name in seen:
        return seen
    seen.add(name)
    for f in re.findall(r'#include "([^"]+\.cuh)"', open(os.path.join(CSRC, name)).read()):
        included(f, seen)
    return seen


def test_the_digest_covers_every_header_of_the_plane_pass():
    files = {os.path.basename(f) for f in bench.PLANE_SOURCES}
    assert included("hpsi2_p.cuh", set()) <= files
    before = bench.kernel_source_digest(bench.PLANE_SOURCES)
    for f in bench.PLANE_SOURCES:
        assert bench.kernel_source_digest([g for g in bench.PLANE_SOURCES if g != f]) != before


def test_a_profile_of_other_sources_gives_no_traffic(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    p = tmp_path / "profiles" / "k.md"
    src = tmp_path / "a.cuh"
    src.write_text("one")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    p.write_text("traffic_bytes_per_launch: 12\nsource_sha256: %s\n" % bench.kernel_source_digest(["a.cuh"]))
    assert bench._profile_traffic("k", ["a.cuh"]) == 12
    src.write_text("two")
    assert bench._profile_traffic("k", ["a.cuh"]) is None
