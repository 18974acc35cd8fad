"""Loops of many bands with an odd number of k-points: the product of the overlaps is a tree, and
a level of an odd number of matrices carries its last one over by a copy of one matrix per loop.
3 and 5 points carry at the first level, 6 only at the second, 7 at both of its odd levels.
Tolerances: N p 2^-47 in the mixed request and 8 sqrt(N p) 2^-52 in FP64, as for loops of 16
points, times ten: the eigenvalue condition numbers over |lambda|, 3 there, reach 22 on these
coarse loops."""
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401
from tests.test_gpu_mixed_many_bands import coupled_copies

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 5, 6, 7])
@pytest.mark.parametrize("copies,precision", [(17, "mixed"), (33, "mixed"), (33, "fp64")])
def test_odd_levels_of_the_product(lib, ctx, copies, precision, N):
    model = coupled_copies(copies, 4)
    plane, p = I.Plane(N, 3, origin=(0.013, 0.021, 0.0)), 2 * copies
    ph, _ = lib.wilson_loop(model, plane, p, precision=precision, ctx=ctx)
    ref, _ = oracle.wilson_loop(model, plane, p)
    tol = N * p * 2.0 ** -47 if precision == "mixed" else 8.0 * (N * p) ** 0.5 * 2.0 ** -52
    assert circ_err_rows(ph.cpu().numpy(), ref) <= 10.0 * tol
