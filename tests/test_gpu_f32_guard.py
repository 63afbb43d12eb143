"""The fault guard's count (bp_get_faults) when changes are not finite: every
weight change that is not a number or out of range counts once, and nothing
else does -- the float32 kernels work on rows padded to 16 bytes (and, on the
cluster, to whole lanes), whose padding columns are not weight changes.

The expected counts are exact.  A NaN input makes every delta of its pattern, so
every change of the group, NaN.  An infinite target makes one output delta and
all hidden deltas infinite: the changes of that output's row (h > 0) and of every
hidden row (infinite or, where the input is 0, NaN).  No change passes the guard,
whose threshold no finite change reaches, so that the weights that would have
taken one keep their bits.
"""
import numpy as np
import pytest

from paper_1801_01554_gb300 import bp, synth
from test_gpu_f32 import dev, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def nonfinite_count(sizes, B, plant):
    X, T, theta = problem(sizes, B, seed=91)
    if plant == "nan input":
        X[B // 2, 3] = np.nan
        bad = np.ones(theta.size, dtype=bool)
    else:
        T[B // 2, 1] = np.inf
        bad = np.zeros(theta.size, dtype=bool)
        offs, _ = synth.param_layout(sizes)
        for l, (wo, bo) in enumerate(offs, start=1):
            rows = [1] if l == len(offs) else range(sizes[l])
            for j in rows:
                bad[wo + j * sizes[l - 1]:wo + (j + 1) * sizes[l - 1]] = True
                bad[bo + j] = True
    with bp.Net(sizes, 0.01, 0.9, bp.BP_F32, max_batch=B) as net:
        net.set_weights(theta)
        net.set_guard(1e30)
        net.train_batch(dev(X), dev(T), B)
        with pytest.raises(bp.BPError) as e:
            net.check()
        assert e.value.status == bp.BP_ENONFINITE
        W, V = net.get_weights(), net.get_velocity()
        np.testing.assert_array_equal(W[bad], theta[bad].astype(np.float32))
        np.testing.assert_array_equal(V[bad], 0.0)
        assert np.isfinite(W).all() and np.isfinite(V).all()
        return net.get_faults(), int(bad.sum())


@pytest.mark.parametrize("plant", ["nan input", "infinite target"])
@pytest.mark.parametrize("sizes", [(203, 120, 26), (202, 61, 26), (17, 9, 3)])
@pytest.mark.parametrize("B", [1, 2, 4])
def test_guard_counts_weight_changes_only_on_the_cluster(sizes, B, plant):
    got, want = nonfinite_count(sizes, B, plant)
    assert got == want


@pytest.mark.parametrize("plant", ["nan input", "infinite target"])
@pytest.mark.parametrize("sizes", [(203, 120, 26), (202, 57, 26), (17, 9, 3)])
def test_guard_counts_weight_changes_only_in_large_groups(sizes, plant):
    got, want = nonfinite_count(sizes, 6200, plant)
    assert got == want


@pytest.mark.parametrize("plant", ["nan input", "infinite target"])
@pytest.mark.parametrize("B", [1, 2, 4])
def test_guard_counts_weight_changes_only_on_one_cta(B, plant):
    got, want = nonfinite_count((64, 33, 17, 9), B, plant)
    assert got == want


@pytest.mark.parametrize("plant", ["nan input", "infinite target"])
@pytest.mark.parametrize("sizes,B", [((203, 120, 26), 512), ((202, 61, 26), 5), ((64, 33, 17, 9), 300)])
def test_guard_counts_weight_changes_only_on_the_grid_wide_kernel(sizes, B, plant):
    got, want = nonfinite_count(sizes, B, plant)
    assert got == want
