"""The fingerprint that decides whether committed profile counts still belong to the stage kernels covers every header that
the kernels' own header includes, so that a change of their arithmetic changes it."""
import os
import re

import bench

CSRC = "paper_2211_16933_gb300/csrc"


def _included(path, seen):
    """Files that `path` includes by quoted name, and what they include."""
    for name in re.findall(r'^\s*#include "([^"]+)"', open(os.path.join(bench.ROOT, path), encoding="utf-8").read(), re.M):
        f = os.path.normpath(os.path.join(os.path.dirname(path), name))
        if not os.path.exists(os.path.join(bench.ROOT, f)):
            f = os.path.join("include", name)  # the compiler's -I
        if f not in seen:
            seen.add(f)
            _included(f, seen)
    return seen


def test_the_fingerprint_covers_the_stage_kernels_headers():
    needed = _included(f"{CSRC}/fdlb_kernels.cuh", set())
    assert f"{CSRC}/qlbm_internal.h" in needed
    for sources in bench._STAGE_SOURCES.values():
        assert needed <= set(sources), needed - set(sources)
