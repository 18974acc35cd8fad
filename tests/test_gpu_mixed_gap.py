"""Direct gaps of the mixed request's four-band kernels (double-float Ritz values).

H(k) is a sum of double-float products (absolute error 2^-47 per unit of sum |t|), its Ritz
matrix sums of four of them, each moving an eigenvalue by as much at most: a bound of
32 x 2^-47 |H| on the difference of two eigenvalues, |H| <= the largest row sum of |t|."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3, 4])
@pytest.mark.parametrize("nested", [False, True])
def test_direct_gap_at_double_float_rounding(lib, ctx, seed, nested):
    rng = np.random.default_rng(seed)
    m = I.bbh(rng.uniform(0.4, 0.6), rng.uniform(0.4, 0.6))
    A = rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4))
    T = 0.025 * (A + A.conj().T)  # a full on-site term: no zero entries, no symmetry
    ii, jj = np.nonzero(np.ones((4, 4)))
    m = I.HoppingList(n=4, R=np.concatenate([m.R, np.zeros((16, 3), np.int32)]), i=np.concatenate([m.i, ii]),
                      j=np.concatenate([m.j, jj]), t=np.concatenate([m.t, T[ii, jj]]), dim=2)
    plane = I.Plane(48, 60, origin=(rng.uniform(), rng.uniform(), 0.0))
    if nested:
        gap = lib.nested_wilson_loop(m, plane, 2, m=1, precision="mixed", ctx=ctx)[3]
    else:
        gap = lib.wilson_loop(m, plane, 2, precision="mixed", ctx=ctx)[1]
    _, ref = oracle.wilson_loop(m, plane, 2)
    norm = np.bincount(m.i, np.abs(m.t)).max()
    assert np.max(np.abs(gap.cpu().numpy() - ref)) <= 32 * 2.0 ** -47 * norm
