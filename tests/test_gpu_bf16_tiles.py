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
