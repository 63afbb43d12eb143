"""Large groups of one-hidden-layer nets, whose sums of changes stay
on chip, against the float64 oracle update by update: both pass widths (64 and
128 patterns), shares that end inside a pass, groups that leave CTAs with fewer rows,
layers that end inside a register block and at the largest numbers of hidden units
that fit, even and odd row pitches; a pending change and the fault guard on this
path; and nets past its limits and a deeper one, which keep the tiled (balanced) weight
phase (test_routes.py says which case runs where).  The bars are test_gpu_f32.py's."""
import numpy as np
import pytest

from oracle import bp_oracle as O
from paper_1801_01554_gb300 import bp
from test_gpu_f32 import dev, problem, stepwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


CASES = [
    ((203, 120, 26), 6100 + 37, 6100), ((203, 120, 26), 20000, 20000), ((203, 60, 26), 20500, 20000),
    ((203, 128, 26), 6500, 6500), ((203, 121, 3), 6200, 6200), ((17, 9, 3), 6300 + 1, 6300), ((40, 33, 40), 6400, 6400),
    ((100, 1, 1), 6080, 6080), ((255, 57, 7), 6100, 6100), ((203, 60, 30, 26), 12500, 12300),
    ((203, 117, 26), 6200, 6200), ((203, 59, 26), 2 * 6200, 6200), ((255, 88, 7), 6100, 6100)]


@pytest.mark.parametrize("sizes,n,mb", CASES)
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


@pytest.mark.parametrize("sizes,B,bar", [((203, 60, 26), 16384, 1.9e-7), ((203, 100, 26), 65536, 1.3e-7),
                                         ((255, 57, 7), 65536, 1.5e-7), ((64, 50, 10), 65536, 9e-8)])
def test_error_of_the_changes_of_large_groups(sizes, B, bar):
    """W_1's change of one update against float64, 2-norm.  Chains of 32 patterns and of 16
    columns measure 1.6e-7, 0.97e-7, 1.1e-7 and 0.65e-7; one chain over a CTA's share and over
    a row, whose roundings grow with the square root of their length, 2.1-2.4e-7, 1.7e-7, 2.1e-7
    and 1.2e-7.  The bars lie between (they are 3 to 6 times 2^-25, the rms of a few roundings)."""
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn(B, sizes[0], device="cuda", generator=g)
    T = (torch.rand(B, sizes[2], device="cuda", generator=g) < 0.3).float()
    n0, H, n2 = sizes
    theta = torch.rand((n0 + 1) * H + (H + 1) * n2, device="cuda", generator=g) * 0.6 - 0.3
    with bp.Net(sizes, 1.0, 0.0, bp.BP_F32, max_batch=B) as net:   # V = 1 * G + 0 * V
        net.set_weights(theta.cpu().numpy())
        net.train_batch(X, T, B)
        net.check()
        V = torch.tensor(net.get_velocity(), device="cuda").double()
    th = theta.double()
    W1, b1, W2 = th[:n0 * H].view(H, n0), th[n0 * H:(n0 + 1) * H], th[(n0 + 1) * H:-n2].view(n2, H)
    h = torch.sigmoid(torch.addmm(b1, X.double(), W1.T))
    o = torch.sigmoid(torch.addmm(th[-n2:], h, W2.T))
    d2 = (T.double() - o) * o * (1 - o)
    ref = (((d2 @ W2) * h * (1 - h)).T @ X.double()).flatten()
    assert float((V[:n0 * H] - ref).norm() / ref.norm()) <= bar


@pytest.mark.parametrize("sizes,n,mb", [((203, 60, 26), 100, 8192), ((203, 60, 26), 2 * 6080 + 1, 6080),
                                        ((64, 50, 10), 6079, 16384), ((203, 120, 26), 6080 + 6079, 6080)])
def test_short_groups_take_the_grid_wide_kernel_step_by_step(sizes, n, mb):
    """Fewer patterns than a pass is worth, in all or in the last group; the first of them
    with a pending change."""
    X, T, theta = problem(sizes, n, seed=44)
    stepwise(sizes, X, T, theta, np.zeros_like(theta), mb, 0.002, 0.9)
    st = O.State(sizes, theta, lr=0.002, momentum=0.9)
    with bp.Net(sizes, 0.002, 0.9, bp.BP_F32, max_batch=mb) as net:
        net.set_weights(theta)
        Xd, Td = dev(X), dev(T)
        net.forward(Xd, 64)
        net.backward(Td, 64)
        net.train_epoch(Xd, Td, n, mb)
        net.check()
        O.backward_accumulate(st, X[:64], T[:64])
        O.train_epoch(st, X, T, mb)
        np.testing.assert_allclose(net.get_weights(), st.theta, rtol=0, atol=1e-5 * np.max(np.abs(st.theta)))
        np.testing.assert_array_equal(net.get_grads(), 0.0)
