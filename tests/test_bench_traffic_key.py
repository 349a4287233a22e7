"""bench.py's key of a traffic capture changes with any source of the headline kernel."""
import os
import re
import shutil

import pytest

import bench


@pytest.mark.parametrize("name", bench.HEADLINE_SOURCES)
def test_key_follows_every_source(tmp_path, name):
    for n in bench.HEADLINE_SOURCES:
        os.makedirs(tmp_path / os.path.dirname(n), exist_ok=True)
        shutil.copy(os.path.join(bench.ROOT, n), tmp_path / n)
    before = bench.source_sha(tmp_path)
    assert before == bench.source_sha()
    with open(tmp_path / name, "a") as f:
        f.write("\n")
    assert bench.source_sha(tmp_path) != before


def test_sources_hold_what_the_kernel_includes():
    """full.cu instantiates the headline kernel; what it includes is in the key."""
    todo, seen = ["paper_2002_11710_gb300/csrc/full.cu"], set()
    while todo:
        n = todo.pop()
        seen.add(n)
        for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(bench.ROOT, n)).read()):
            path = os.path.join(os.path.dirname(n), inc)
            path = path if os.path.exists(os.path.join(bench.ROOT, path)) else os.path.join("include", inc)
            if path not in seen:
                todo.append(path)
    assert seen <= set(bench.HEADLINE_SOURCES)
