"""bench.py takes the committed ncu counters for the sources they were measured
on: the digest covers every file that the sweep kernels are compiled from."""

import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2108_07549_gb300", "csrc")


def test_digest_covers_every_included_file(monkeypatch, tmp_path):
    seen, todo = set(), ["sweep.cu"]
    while todo:
        name = todo.pop()
        if name in seen or not os.path.exists(os.path.join(CSRC, name)):
            continue
        seen.add(name)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read())
    target = tmp_path / "paper_2108_07549_gb300" / "csrc"
    target.mkdir(parents=True)
    for name in seen:
        (target / name).write_bytes(open(os.path.join(CSRC, name), "rb").read())
    want = bench.source_digest()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.source_digest() == want
    for name in sorted(seen):
        with open(target / name, "ab") as fh:
            fh.write(b"\n")
        changed = bench.source_digest()
        assert changed != want, name
        want = changed
