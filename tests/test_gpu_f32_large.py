"""Large groups of one-hidden-layer nets, whose sums of changes stay in
registers, against the float64 oracle update by update: both pass widths (64 and
128 patterns), shares that end inside a pass, a ragged last group that leaves
CTAs without patterns, layers that end inside a register block, even and odd row
pitches; a pending change and the fault guard on this path; and a deeper net,
which keeps the tiled (balanced) weight phase.  The bars are test_gpu_f32.py's."""
import numpy as np
import pytest

from oracle import bp_oracle as O
from paper_1801_01554_gb300 import bp
from test_gpu_f32 import dev, problem, stepwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,n,mb", [
    ((203, 120, 26), 6100 + 37, 6100), ((203, 120, 26), 20000, 20000), ((203, 60, 26), 20500, 20000),
    ((203, 128, 26), 6500, 6500), ((203, 121, 3), 6200, 6200), ((17, 9, 3), 6300 + 1, 6300), ((40, 33, 40), 6400, 6400),
    ((100, 1, 1), 6080, 6080), ((255, 57, 7), 6100, 6100), ((203, 60, 30, 26), 12500, 12300)])
def test_large_groups_match_oracle_step_by_step(sizes, n, mb):
    X, T, theta = problem(sizes, n, seed=41)
    stepwise(sizes, X, T, theta, np.zeros_like(theta), mb, 0.002, 0.9)


def test_pending_change_and_guard_on_large_groups():
    sizes, B = (203, 60, 26), 6200
    X, T, theta = problem(sizes, B, seed=42)
    st = O.State(sizes, theta, lr=0.002, momentum=0.9)
    with bp.Net(sizes, 0.002, 0.9, bp.BP_F32, max_batch=B) as net:
        net.set_weights(theta)
        Xd, Td = dev(X), dev(T)
        net.forward(Xd, B)
        net.backward(Td, B)
        net.train_batch(Xd, Td, B)
        net.check()
        O.backward_accumulate(st, X, T)
        O.train_batch(st, X, T)
        np.testing.assert_allclose(net.get_weights(), st.theta, rtol=0, atol=1e-5 * np.max(np.abs(st.theta)))
        np.testing.assert_array_equal(net.get_grads(), 0.0)
        w = net.get_weights()
        net.set_velocity(np.zeros_like(theta))
        net.set_guard(1e-30)   # every change that is not zero is out of range
        net.train_batch(Xd, Td, B)
        net.check()
        np.testing.assert_array_equal(net.get_weights(), w)
        assert net.get_faults() > 0.9 * theta.size
