"""A scan of more loops than 32-bit thread indices of a warp per loop reach (2^27)."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu


def test_more_than_2_27_loops(lib):
    import torch
    if torch.cuda.get_device_properties(0).total_memory < 64 << 30:
        pytest.skip("needs 20 GB of states and gaps")
    Nt = 2 ** 27 + 3
    model, origin = I.chern_eq4(1.3), (0.11, 0.23, 0.0)
    c = lib.Context(0)
    try:
        ph, gap = lib.wilson_loop(model, I.Plane(3, Nt, origin=origin), 1, precision="fp64", ctx=c)
        for i in (0, 1, 2 ** 27 - 1, 2 ** 27, 2 ** 27 + 1, 2 ** 27 + 2):
            ref, rgap = oracle.wilson_loop(model, I.Plane(3, 1, origin=(origin[0], origin[1] + i / Nt, 0.0)), 1)
            assert abs(np.angle(np.exp(1j * (float(ph[i, 0]) - ref[0, 0])))) <= 1e-10, i
            assert abs(float(gap[i]) - rgap[0]) <= 1e-10, i
    finally:
        c.close()
