"""The benchmark names the launch shape that the library uses: a lane per
half-word of 32 trees, up to a warp; the knob counts for twice that only."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class _Tuned:
    def __init__(self, words, group):
        self.knobs = {"bfs_words": words, "bfs_group": group}

    def get_tuning(self):
        return self.knobs


@pytest.mark.parametrize("words,group,want", [(0, 0, (32, 32)), (32, 32, (32, 32)), (16, 0, (16, 32)), (16, 16, (16, 32)),
                                              (8, 0, (8, 16)), (8, 32, (8, 32)), (8, 8, (8, 16)), (4, 32, (4, 8)),
                                              (1, 0, (1, 2)), (1, 4, (1, 4)), (5, 0, (5, 16))])
def test_bfs_shape_follows_the_library(words, group, want):
    spec = importlib.util.spec_from_file_location("bench_shape_under_test", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    assert bench.bfs_shape(_Tuned(words, group)) == want
