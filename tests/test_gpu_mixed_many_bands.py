"""Mixed request with many occupied bands: the loop products in double-float and the
eigenphases (FP64 up to 127 bands, double-float on a cluster beyond).

Weakly coupled copies of gapped four-band models: the Wilson matrix is close to a direct sum of
2 x 2 blocks, its eigenphases are well conditioned, and the FP32 seed's error squared stays
below the double-float roundings.  Those move a phase by about one unit 2^-47 per product and
band at most: N p 2^-47."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu


def coupled_copies(copies, seed, eps=1e-3):
    """Copies with random couplings, on-site shifts within +-0.3 and a random Hermitian
    on-site coupling of size eps."""
    rng = np.random.default_rng(seed)
    m = I.direct_sum([I.bbh(rng.uniform(0.4, 0.6), rng.uniform(0.4, 0.6)) if c % 2
                      else I.spin_hall(rng.uniform(0.8, 1.2)) for c in range(copies)])
    n = m.n
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    T = eps * 0.5 * (A + A.conj().T) + np.diag(np.repeat(0.3 * rng.uniform(-1, 1, copies), 4))
    ii, jj = np.nonzero(np.ones((n, n)))
    return I.HoppingList(n=n, R=np.concatenate([m.R, np.zeros((n * n, 3), np.int32)]),
                         i=np.concatenate([m.i, ii]), j=np.concatenate([m.j, jj]),
                         t=np.concatenate([m.t, T[ii, jj]]), dim=2)


@pytest.mark.parametrize("copies,seed", [(24, 1), (40, 1), (40, 2), (72, 1), (72, 2)])
def test_mixed_phases_at_double_float_rounding(lib, ctx, copies, seed):
    model = coupled_copies(copies, seed)
    plane, p = I.Plane(16, 12, origin=(0.013, 0.021, 0.0)), 2 * copies
    ph, _ = lib.wilson_loop(model, plane, p, precision="mixed", ctx=ctx)
    ref, _ = oracle.wilson_loop(model, plane, p)
    assert circ_err_rows(ph.cpu().numpy(), ref) <= plane.N * p * 2.0 ** -47


@pytest.mark.parametrize("copies", [17, 63, 64])
def test_mixed_phases_at_the_solvers_limits(lib, ctx, copies):
    # p = 34 (the first beyond one CTA per loop) and 126: FP64 eigenphases; 128: double-float
    model = coupled_copies(copies, 3)
    plane, p = I.Plane(9, 3, origin=(0.013, 0.021, 0.0)), 2 * copies
    ph, _ = lib.wilson_loop(model, plane, p, precision="mixed", ctx=ctx)
    ref, _ = oracle.wilson_loop(model, plane, p)
    assert circ_err_rows(ph.cpu().numpy(), ref) <= plane.N * p * 2.0 ** -47


@pytest.mark.parametrize("copies,seed", [(16, 6), (24, 1), (24, 3), (40, 1), (40, 7)])
def test_fp64_phases_at_rounding(lib, ctx, copies, seed):
    # the same in FP64: units of 2^-52 from N p independent roundings, with a factor of eight
    # (8 sqrt(N p) 2^-52).  With a weak coupling many entries next to the diagonal of the
    # Hessenberg matrix are small at once
    model = coupled_copies(copies, seed, eps=1e-4)
    plane, p = I.Plane(16, 24, origin=(0.013, 0.021, 0.0)), 2 * copies
    ph, _ = lib.wilson_loop(model, plane, p, precision="fp64", ctx=ctx)
    ref, _ = oracle.wilson_loop(model, plane, p)
    assert circ_err_rows(ph.cpu().numpy(), ref) <= 8 * np.sqrt(plane.N * p) * 2.0 ** -52
