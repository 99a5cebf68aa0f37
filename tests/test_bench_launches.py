"""What bench.py says about the engine's launches and tile lists is what the sources say."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _source(name):
    return open(os.path.join(ROOT, "paper_2606_21791_gb300", "csrc", name)).read()


@pytest.mark.parametrize("variants,views", [(127, 4), (128, 4), (2048, 4), (8192, 4), (511, 1), (512, 1), (32, 16)])
def test_launches_per_step(variants, views):
    import bench
    at = int(re.search(r"constexpr int kSortPairs = (\d+);", _source("k_blend.cu")).group(1))
    assert bench.launches_per_step(variants, views) == (6 if variants * views >= at else 4)


def test_grids_listed_by_counting():
    import bench
    assert bench.DIRECT_TILES == int(re.search(r"return nt <= (\d+) \|\|", _source("k_sort.cu")).group(1))
