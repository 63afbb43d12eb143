"""Which kernel a float32 training call runs on, as the library decides it from the
sizes (test infrastructure; host code, no GPU)."""
import ctypes

from paper_1801_01554_gb300 import bp

CLUSTER, ONE_CTA, LARGE, GRID = "cluster", "one CTA", "large", "grid"


def route(sizes, minibatch, n=None, pending=False, num_sms=152):
    f = bp.load().bp_internal_f32_route
    arr = (ctypes.c_int * len(sizes))(*sizes)
    k = f(arr, len(sizes), int(minibatch), int(minibatch if n is None else n), num_sms, int(pending))
    return [CLUSTER, ONE_CTA, LARGE, GRID][k]
