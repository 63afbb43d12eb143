"""bfloat16 path at the edges of its tiles: K-major and MN-major operands whose
rows, columns and batch end inside a 64-wide block, every tile width (64, 128
and 256 columns) and pooled changes cut into several K splits.

Tolerance as in test_gpu_bf16.py (2e-2 normwise per layer: inputs, weight
copies, activations and deltas rounded to bfloat16, fp32 accumulation); a
misplaced operand block is an error of order one.
"""
import numpy as np
import pytest

from oracle import bp_oracle as O
from paper_1801_01554_gb300 import bp
from parity import assert_layers, normwise
from test_gpu_bf16 import TOL, dev_bf16, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [((8, 8, 8), 1), ((72, 264, 136), 129), ((320, 520, 64), 63), ((136, 1032, 40), 127),
         ((64, 128, 32), 4100), ((256, 328, 200, 72), 1025), ((256, 512, 64), 20000),
         ((136, 2312, 264), 130)]   # more than one group of row blocks in the pooled changes


@pytest.mark.parametrize("sizes,B", CASES)
def test_step_at_tile_edges_matches_oracle(sizes, B):
    X, T, theta = problem(sizes, B, seed=B)
    st = O.State(sizes, theta, lr=0.01, momentum=0.9, grad_scale=1.0 / B)
    As, _, G_ref, e_ref = O.step_quantities(st, X, T)
    Xd, Td = dev_bf16(X), dev_bf16(T)
    Yd = torch.empty((B, sizes[-1]), dtype=torch.bfloat16, device="cuda")
    sse = torch.zeros(2, device="cuda")
    with bp.Net(sizes, 0.01, 0.9, bp.BP_BF16, max_batch=B, grad_scale=1.0 / B) as net:
        net.set_weights(theta)
        net.forward(Xd, B, Yd)
        net.backward(Td, B, sse[:1])
        net.check()
        G = net.get_grads()
    with bp.Net(sizes, 0.01, 0.9, bp.BP_BF16, max_batch=B, grad_scale=1.0 / B) as net:
        net.set_weights(theta)
        net.train_batch(Xd, Td, B, sse[1:])
        net.check()
        th = net.get_weights()
    assert normwise(Yd.float().cpu().numpy(), As[-1]) <= TOL
    np.testing.assert_allclose(sse.cpu().numpy(), [e_ref, e_ref], rtol=TOL)
    assert_layers(sizes, G, G_ref, TOL, None, "G")
    st.G = G_ref
    O.apply_update(st)
    assert_layers(sizes, th - theta, st.theta - theta, TOL, None, "W1-W0")


@pytest.mark.parametrize("sizes,B", [((208, 520, 64), 300), ((64, 128, 32), 4100)])
def test_pending_change_is_folded_into_train_batch(sizes, B):
    """Update in the pooled change's epilogue, and in the kernel after split sums."""
    X, T, theta = problem(sizes, B, seed=51)
    X2, T2, _ = problem(sizes, B, seed=52)
    st = O.State(sizes, theta, lr=0.01, momentum=0.9, grad_scale=1.0 / B)
    with bp.Net(sizes, 0.01, 0.9, bp.BP_BF16, max_batch=B, grad_scale=1.0 / B) as net:
        net.set_weights(theta)
        Xd, X2d = dev_bf16(X), dev_bf16(X2)
        for k in range(2):   # the second step has a velocity
            net.forward(Xd, B)
            net.backward(dev_bf16(T), B)
            net.train_batch(X2d, dev_bf16(T2), B)
            O.backward_accumulate(st, X, T)
            O.train_batch(st, X2, T2)
        net.check()
        th, V = net.get_weights(), net.get_velocity()
        np.testing.assert_array_equal(net.get_grads(), 0.0)
    assert_layers(sizes, th - theta, st.theta - theta, TOL, None, "W2-W0")
    assert_layers(sizes, V, st.V, TOL, None, "V2")


def one_step_change(sizes, B, seed):
    """One update with lr 1, momentum 0: V is the pooled change.  Returns V, the change that
    bp_backward leaves in G, the outputs, and X, T, theta, all on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(B, sizes[0], device="cuda", generator=g).bfloat16()
    T = (torch.rand(B, sizes[-1], device="cuda", generator=g) < 0.3).bfloat16()
    theta = torch.cat([torch.cat([torch.randn(i * o, device="cuda", generator=g) / i ** 0.5,
                                  torch.rand(o, device="cuda", generator=g) * 0.2 - 0.1])
                       for i, o in zip(sizes[:-1], sizes[1:])])
    Y = torch.empty(B, sizes[-1], dtype=torch.bfloat16, device="cuda")
    with bp.Net(sizes, 1.0, 0.0, bp.BP_BF16, max_batch=B) as net:
        net.set_weights(theta.cpu().numpy())
        net.forward(X, B, Y)
        net.backward(T, B)
        net.check()
        G = torch.tensor(net.get_grads(), device="cuda")
    with bp.Net(sizes, 1.0, 0.0, bp.BP_BF16, max_batch=B) as net:
        net.set_weights(theta.cpu().numpy())
        net.train_batch(X, T, B)
        net.check()
        V = torch.tensor(net.get_velocity(), device="cuda")
    return V, G, Y, X, T, theta


@pytest.mark.parametrize("sizes,B,chain", [((208, 1024), 512, 192), ((1024, 2048), 1001, 512),
                                           ((1024, 2048), 8192, 4096), ((4096, 4096), 16384, 8192)])
def test_pooled_change_error_is_that_of_its_chains(sizes, B, chain):
    """Sums of the change of one layer against float64 sums of the same bf16 deltas and
    inputs.  The tensor cores truncate as they accumulate, 16 patterns a step: a running sum of
    random signs, on average 2/3 of its end, loses up to an ulp (2^-23, half of it on
    average) a step, 1.8e-9 of the end per pattern of the chain.  Measured: 0.7 to 1.04e-9; the
    bar is 1.3e-9 times the chain (1.2e-5, 5.3e-6, 6.7e-7, 2.5e-7), which one chain over the
    batch exceeds (1.7e-5, 8.0e-6, 7.4e-7, 3.4e-7)."""
    V, G, Y, X, T, _ = one_step_change(sizes, B, seed=1)
    o = Y.float()
    d = ((T.float() - o) * o * (1 - o)).bfloat16().double()
    ref = (d.T @ X.double()).flatten()
    nw = ref.numel()
    for got in (V, G):
        err = float((got[:nw].double() - ref).norm() / ref.norm())
        assert err <= 1.3e-9 * chain, err


@pytest.mark.parametrize("sizes,B,alike", [((4096, 4096, 64), 8192, True), ((1024, 1024, 32), 4096, False),
                                           ((2048, 1024, 8), 4096, False)])
def test_chains_of_two_layers_in_one_launch(sizes, B, alike):
    """Tiles of 256 columns with two and eight chains (the accumulators take turns), of 64 with
    four and eleven and of 128 with two and eleven (more than there are accumulators), against
    float64; in the first bp_backward has the same tiles and sums alike, bit for bit."""
    V, G, _, X, T, theta = one_step_change(sizes, B, seed=2)
    assert not alike or torch.equal(V, G)
    nw = sizes[0] * sizes[1]
    W1, b1 = theta[:nw].view(sizes[1], sizes[0]).double(), theta[nw:nw + sizes[1]].double()
    W2 = theta[nw + sizes[1]:-sizes[2]].view(sizes[2], sizes[1]).double()
    h = torch.sigmoid(torch.addmm(b1, X.double(), W1.T))
    o = torch.sigmoid(torch.addmm(theta[-sizes[2]:].double(), h, W2.T))
    d2 = (T.double() - o) * o * (1 - o)
    d1 = (d2 @ W2) * h * (1 - h)
    for C in (V, G):
        for got, ref in ((C[:nw], d1.T @ X.double()), (C[nw + sizes[1]:-sizes[2]], d2.T @ h)):
            assert normwise(got.double().cpu().numpy(), ref.flatten().cpu().numpy()) <= TOL


@pytest.mark.parametrize("n,B,shift", [(2048, 8192, 0), (768, 20000, 0), (512, 20000, 640)])
def test_forward_of_one_layer_may_write_over_its_input(n, B, shift):
    """Y may be X itself, or overlap it by rows (a square one-layer net), also where the tiles
    of a row block run in different waves: the outputs of a call with a buffer of its own."""
    X, _, theta = problem((n, n), B, seed=53)
    buf = torch.zeros((B + shift, n), dtype=torch.bfloat16, device="cuda")
    buf[:B] = dev_bf16(X)
    Y = torch.empty((B, n), dtype=torch.bfloat16, device="cuda")
    with bp.Net((n, n), 0.01, 0.9, bp.BP_BF16, max_batch=B) as net:
        net.set_weights(theta)
        net.forward(buf[:B], B, Y)
        net.forward(buf[:B], B, buf[shift:])
        net.check()
    assert torch.equal(buf[shift:], Y)
