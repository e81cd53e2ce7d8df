"""bench.py reports a recorded traffic figure only while the rollout's sources are those it was
taken on: the digest covers every source that the rollout's kernels are compiled from."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_02869_gb300", "csrc")


def _sources(name, seen):
    """`name` and what it includes of its own folder (the public header beside it is the interface)."""
    if name in seen or "/" in name or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'#include "([^"]+)"', f.read()):
            _sources(inc, seen)
    return seen


def test_digest_covers_the_rollouts_sources():
    want = _sources("rollout.cu", set()) | _sources("rollout_traj.cu", set())
    assert "wind_rollout.cuh" in want
    assert want <= set(bench.ROLLOUT_SOURCES), want - set(bench.ROLLOUT_SOURCES)


def test_digest_follows_every_source(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_1506_02869_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in bench.ROLLOUT_SOURCES:
        (csrc / f).write_text(f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    seen = {bench.rollout_sources_digest()}
    for f in bench.ROLLOUT_SOURCES:
        (csrc / f).write_text(f + " changed")
        seen.add(bench.rollout_sources_digest())
    assert len(seen) == 1 + len(bench.ROLLOUT_SOURCES)
