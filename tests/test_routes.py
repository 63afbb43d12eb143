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
