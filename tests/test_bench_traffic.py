"""The roofline's DRAM figure is dropped when any source that decides it has changed (no GPU)."""
import hashlib
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

SOURCES = [bench.STAGE_SRC, *bench.STAGE_PARTS]


def _summary(tmp_path, files):
    sha = [hashlib.sha256(b"".join(open(f, "rb").read() for f in fs)).hexdigest() for fs in (files[:1], files[1:])]
    p = tmp_path / "p.md"
    p.write_text(f"stage kernel source sha256: {sha[0]}\nincluded sources sha256 (a, b): {sha[1]}\nstage variant: 1\n"
                 "dram bytes per launch (read + write): 4.9e7\n")
    return str(p)


@pytest.mark.parametrize("changed", [None, *range(len(SOURCES))])
def test_a_change_in_any_source_drops_the_figure(tmp_path, monkeypatch, changed):
    copies = []
    for k, f in enumerate(SOURCES):
        c = tmp_path / os.path.basename(f)
        c.write_bytes(open(f, "rb").read() + (b"//\n" if k == changed else b""))
        copies.append(str(c))
    monkeypatch.setattr(bench, "PROFILE_SUMMARY", _summary(tmp_path, SOURCES))
    monkeypatch.setattr(bench, "STAGE_SRC", copies[0])
    monkeypatch.setattr(bench, "STAGE_PARTS", copies[1:])
    assert bench.recorded_traffic(1) == (4.9e7 if changed is None else None)


def test_the_committed_summary_names_every_source():
    text = open(bench.PROFILE_SUMMARY).read()
    line = next(x for x in text.splitlines() if x.startswith("included sources sha256"))
    assert all(os.path.basename(f) in line for f in bench.STAGE_PARTS)
    assert os.path.basename(bench.STAGE_SRC) == "dg_stage.cuh" and "stage kernel source sha256:" in text
