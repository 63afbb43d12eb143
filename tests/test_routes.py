"""The float32 training kernel of a call, by its sizes (CPU: the rule is host code)."""
import os

import pytest

from paper_1801_01554_gb300 import bp
from routes import CLUSTER, GRID, LARGE, ONE_CTA, route


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not os.path.exists(bp.lib_path()):
        from paper_1801_01554_gb300 import build
        build.build()


@pytest.mark.parametrize("sizes,mb,n,want", [
    ((203, 120, 26), 6080, 6080, LARGE), ((203, 120, 26), 6079, 65536, GRID),
    # the group, not the argument: too few patterns for a pass of the large-group kernel
    ((203, 60, 26), 8192, 100, GRID), ((203, 60, 26), 8192, 6079, GRID), ((203, 60, 26), 8192, 6080, LARGE),
    ((203, 60, 26), 8192, 8192 + 100, LARGE)])   # (its last group goes to the grid-wide kernel)
def test_large_groups_by_the_patterns_there_are(sizes, mb, n, want):
    assert route(sizes, mb, n) == want


@pytest.mark.parametrize("sizes,mb,want", [
    # tests/test_gpu_f32.py
    ((203, 120, 26), 1, CLUSTER), ((203, 60, 26), 3, CLUSTER), ((5, 3, 2), 1, CLUSTER), ((64, 33, 17, 9), 1, ONE_CTA),
    ((64, 33, 17, 9), 4, ONE_CTA), ((40, 300, 200, 1), 2, GRID), ((7, 9, 5, 11, 6, 8, 4, 10, 3), 2, ONE_CTA),
    ((203, 120, 26), 512, GRID), ((203, 120, 26), 16384, LARGE), ((203, 60, 26), 12288, LARGE),
    ((203, 60, 30, 26), 12288, GRID), ((20, 8, 6, 3), 12500, GRID), ((203, 128, 26), 12288, GRID),
    # tests/test_gpu_f32_cluster.py
    ((203, 120, 26), 4, CLUSTER), ((203, 120, 26), 5, GRID), ((203, 300, 26), 1, CLUSTER), ((203, 300, 26), 4, CLUSTER),
    ((203, 250, 26), 2, CLUSTER), ((3, 1, 1), 2, CLUSTER), ((17, 9, 3), 4, CLUSTER), ((15, 33, 5), 3, CLUSTER),
    ((16, 57, 7), 4, CLUSTER), ((895, 90, 3), 2, CLUSTER), ((896, 20, 4), 2, ONE_CTA), ((511, 40, 100), 1, CLUSTER),
    ((40, 20, 128), 1, CLUSTER), ((40, 20, 128), 2, ONE_CTA), ((40, 20, 129), 1, ONE_CTA),
    # tests/test_gpu_f32_large.py
    ((203, 120, 26), 6100, LARGE), ((203, 121, 3), 6200, GRID), ((203, 117, 26), 6200, LARGE), ((203, 59, 26), 6200, LARGE),
    ((17, 9, 3), 6300, LARGE), ((40, 33, 40), 6400, LARGE), ((100, 1, 1), 6080, LARGE), ((255, 57, 7), 6100, LARGE),
    ((255, 88, 7), 6100, LARGE), ((255, 89, 7), 6100, GRID), ((203, 100, 26), 65536, LARGE), ((64, 50, 10), 65536, LARGE)])
def test_the_kernel_that_each_gpu_test_is_named_for(sizes, mb, want):
    assert route(sizes, mb) == want


def test_a_pending_change_keeps_small_groups_on_the_grid_wide_kernel():
    assert route((203, 120, 26), 2, pending=True) == route((64, 33, 17, 9), 2, pending=True) == GRID
    assert route((203, 120, 26), 8192, pending=True) == LARGE
