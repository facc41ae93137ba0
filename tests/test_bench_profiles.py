"""bench.py prints the DRAM traffic of a committed ncu summary only beside a run
that the summary describes: the kernel's current sources and, for the search
kernel, the same cells and schedule (how often lists are read again depends on
both)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

OFF = 0xFFFFFFFF


def _note(tmp_path, schedule):
    sources = ("hc_join.cu", "hc_internal.cuh")
    text = f"    traffic_bytes_per_launch: 123456\n    source_sha256: {bench.source_hash(sources)}\n"
    for s in [schedule] if isinstance(schedule, str) else schedule or []:
        text += f"    schedule: {s}\n"
    path = tmp_path / "note.md"
    path.write_text(text)
    return str(path)


@pytest.mark.parametrize("args,name", [(([64, 1, 1], 16, OFF, 1), "shares 64x1x1, item grain 16, merge off"),
                                       (([64, 1, 1], 0, 0, 0), "shares 64x1x1, item grain by size, merge auto"),
                                       (([16, 4, 1], 64, 32, 4), "shares 16x4x1, item grain 64, merge 32,4")])
def test_traffic_belongs_to_the_schedule(tmp_path, args, name):
    assert bench.schedule_name(*args) == name
    note = _note(tmp_path, name)
    assert bench.profiled_traffic(note, schedule=name) == 123456
    other = bench.schedule_name(args[0], 256, *args[2:])
    assert bench.profiled_traffic(note, schedule=other) is None
    assert bench.profiled_traffic(_note(tmp_path, None), schedule=name) is None
    both = _note(tmp_path, [other, name])  # two names of one launch
    assert bench.profiled_traffic(both, schedule=name) == bench.profiled_traffic(both, schedule=other) == 123456
    note = _note(tmp_path, name)
    assert bench.profiled_traffic(note) == 123456  # a kernel with one schedule names none
