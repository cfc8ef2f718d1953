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


@pytest.mark.parametrize("words,group,K,want", [
    (0, 0, 4096, (32, 32)), (32, 32, 4096, (32, 32)), (16, 0, 4096, (16, 32)), (16, 16, 4096, (16, 32)),
    (0, 0, 1024, (16, 32)), (32, 0, 1024, (16, 32)), (8, 0, 1024, (8, 16)), (8, 32, 1024, (8, 32)), (8, 8, 1024, (8, 16)),
    (4, 32, 1024, (4, 8)), (0, 0, 1, (1, 2)), (1, 4, 4096, (1, 4)), (0, 0, 300, (5, 16))])
def test_bfs_shape_follows_the_library(words, group, K, want):
    spec = importlib.util.spec_from_file_location("bench_shape_under_test", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    assert bench.bfs_shape(_Tuned(words, group), K) == want
