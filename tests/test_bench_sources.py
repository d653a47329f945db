"""The hash that keys the committed profiles covers every sampling kernel's sources."""

import os
import re

import bench
from paper_2503_20566_gb300 import build

CSRC = os.path.join(os.path.dirname(bench.__file__), "paper_2503_20566_gb300", "csrc")


def _closure(name, seen):
    if name not in seen:
        seen.add(name)
        with open(os.path.join(CSRC, name)) as f:
            for inc in re.findall(r'^\s*#include\s+"([^"]+)"', f.read(), flags=re.M):
                _closure(inc, seen)
    return seen


def test_every_kernel_unit_and_header_is_hashed(monkeypatch):
    units = [u for u in build.SOURCES if u.startswith("vmc_")]
    files = set().union(*(_closure(u, set()) for u in units))
    assert files == set(bench.KERNEL_SOURCES) | set(bench.OTHER_UNITS)
    real, before = open, bench.source_hash()
    for name in files:
        class Changed:
            def __init__(self, path, mode="r"):
                self.f, self.extra = real(path, mode), b" " if path.endswith(os.sep + name) else b""

            def __enter__(self):
                return self

            def __exit__(self, *a):
                self.f.close()

            def read(self):
                return self.f.read() + self.extra

        monkeypatch.setattr("builtins.open", Changed)
        after = bench.source_hash()
        monkeypatch.undo()
        assert after != before, name
