"""The bench reports the layer kernels' captured traffic and instructions only
while the sources that they compile from hash to the captured value: the
hashed list is every file of the tree that ara_layer.cu includes."""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1501_06326_gb300", "csrc")


def _included(name, seen):
    if name in seen:
        return seen
    seen.add(name)
    with open(os.path.join(CSRC, name)) as fh:
        for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', fh.read(), re.M):
            _included(inc, seen)
    return seen


def test_layer_sources_are_what_the_layer_kernels_include():
    import bench

    assert set(bench.LAYER_SOURCES) == _included("ara_layer.cu", set())
