"""The bench's roofline of the n > 32 stages: each against the pipe it runs on, and the FP64 request
that starts from an FP32 solve (an lg_polish stage) with its refinement and polish counted."""
import pytest

import bench


@pytest.mark.parametrize("stage,mixed,polished,p,pipe", [
    ("lg_tridiag", True, False, 64, "fp32"), ("lg_tridiag", False, True, 64, "fp32"),
    ("lg_tridiag", False, False, 64, "fp64"), ("lg_refine", False, True, 64, "fp32"),
    ("lg_polish", False, True, 64, "fp64"), ("overlaps", True, False, 200, "fp32"),
    ("overlaps", False, True, 200, "fp64"), ("loops", False, True, 64, "fp64"),
    ("eigenphases", True, False, 64, "fp64"), ("eigenphases", True, False, 200, "fp32"),
    ("eigenphases", False, True, 200, "fp64"),
])
def test_stage_pipe(stage, mixed, polished, p, pipe):
    assert bench.stage_pipe(stage, mixed, polished, p) == pipe
    assert pipe in bench.PIPE_SOURCE


def test_polished_request_counts_refinement_and_polish():
    n, p, N, Nt = 256, 64, 101, 101
    K = N * Nt
    fl = bench.manyband_stage_flops(n, p, N, Nt, 1000, False, n * n, polished=True)
    mixed = bench.manyband_stage_flops(n, p, N, Nt, 1000, True, n * n)
    assert fl["lg_refine"] == mixed["lg_refine"]
    assert fl["lg_backtransform"] == mixed["lg_backtransform"]
    # H Q, half of Q^dag (H Q), Q G, half of Q^dag Q: 8 real flops per complex multiply-add
    assert fl["lg_polish"] == pytest.approx(K * 8.0 * (n * n * p + n * p * p / 2 + n * p * p + n * p * p / 2))
