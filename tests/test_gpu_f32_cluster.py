"""Groups of up to 4 patterns of one-hidden-layer nets on one cluster, against the
float64 oracle update by update: every group size, ragged groups, 1 to 8 CTAs, CTAs without
units, both row splits (4 and 7 float4 columns a lane) and the widest output
layer (128 outputs, groups of 1); and the nets and groups just past the limits, which other
kernels take (test_routes.py says which case runs where).  The bars
are test_gpu_f32.py's (1e-5 of each sum's magnitude, plus the roundings of the
stored weight changes)."""
import numpy as np
import pytest

from paper_1801_01554_gb300 import bp, synth
from test_gpu_f32 import problem, stepwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


CASES = [
    ((203, 120, 26), 23, 4, 0.05), ((203, 120, 26), 65, 3, 0.05), ((203, 120, 26), 70, 5, 0.05),
    ((203, 300, 26), 30, 1, 0.05), ((203, 300, 26), 45, 4, 0.05), ((203, 250, 26), 21, 2, 0.05),
    ((3, 1, 1), 9, 2, 0.05), ((17, 9, 3), 41, 4, 0.05), ((15, 33, 5), 33, 3, 0.05), ((16, 57, 7), 40, 4, 0.05),
    ((895, 90, 3), 12, 2, 0.02), ((511, 40, 100), 9, 1, 0.02), ((40, 20, 128), 10, 2, 0.02),
    ((896, 20, 4), 6, 2, 0.02), ((40, 20, 129), 6, 1, 0.02), ((203, 120, 26), 40, 17, 0.05),
    ((40, 20, 128), 7, 1, 0.02)]


@pytest.mark.parametrize("sizes,n,mb,lr", CASES)
def test_cluster_groups_match_oracle_step_by_step(sizes, n, mb, lr):
    X, T, theta = problem(sizes, n, seed=31)
    V0 = synth.round_to(np.random.default_rng(4).uniform(-1e-3, 1e-3, theta.size), "f32")
    stepwise(sizes, X, T, theta, V0, mb, lr, 0.9)


@pytest.mark.parametrize("mb", [1, 4])
def test_cluster_groups_with_the_table_logistic(mb):
    sizes, n = (203, 60, 26), 29
    X, T, theta = problem(sizes, n, seed=32)
    stepwise(sizes, X, T, theta, np.zeros_like(theta), mb, 0.05, 0.9, squash="table")


def test_cluster_groups_report_a_nonfinite_error_sum():
    sizes, n = (40, 16, 5), 12
    X, T, theta = problem(sizes, n, seed=33)
    X[7, 3] = np.nan
    with bp.Net(sizes, 0.05, 0.9, bp.BP_F32, max_batch=4) as net:
        net.set_weights(theta)
        net.train_epoch(torch.tensor(X, dtype=torch.float32, device="cuda"),
                        torch.tensor(T, dtype=torch.float32, device="cuda"), n, 4)
        with pytest.raises(bp.BPError) as e:
            net.check()
        assert e.value.status == bp.BP_ENONFINITE


@pytest.mark.parametrize("sizes,n,mb", [((203, 60, 26), 41, 3), ((203, 60, 26), 70, 4), ((64, 33, 17, 9), 21, 2)])
def test_noalloc_small_groups_match_bp_train_epoch(sizes, n, mb):
    """The same kernels on the caller's buffers: the same bits."""
    X, T, theta = problem(sizes, n, seed=34)
    Xd = torch.tensor(X, dtype=torch.float32, device="cuda")
    Td = torch.tensor(T, dtype=torch.float32, device="cuda")
    sse = torch.zeros(2, -(-n // mb), device="cuda")
    th = torch.tensor(theta, dtype=torch.float32, device="cuda")
    V = torch.zeros_like(th)
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    with bp.Net(sizes, 0.05, 0.9, bp.BP_F32, max_batch=mb) as net:
        net.set_weights(theta)
        for _ in range(2):
            net.train_epoch(Xd, Td, n, mb, sse[0])
            bp.bp_train_epoch_noalloc(sizes, 0.05, 0.9, 1.0, th, V, Xd, Td, n, mb, sse[1], status)
        net.check()
        np.testing.assert_array_equal(th.cpu().numpy(), net.get_weights())
        np.testing.assert_array_equal(V.cpu().numpy(), net.get_velocity())
    np.testing.assert_array_equal(sse[0].cpu().numpy(), sse[1].cpu().numpy())
    assert status.item() == 0
