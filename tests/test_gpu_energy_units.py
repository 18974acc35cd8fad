"""FP64 requests do not depend on the unit of energy, nor on a level far from the band edge: the
FP32 solve they may start from sees H in units of its largest hopping, and k-points that the
FP64 corrections cannot take (a gap below 1e-3 of the spectral radius, band edges of more
than eight levels) are solved in FP64.  Phases within 1e-10 of the oracle, gaps within 8 n eps
|H| (the forward error of a backward-stable eigenvalue, with a factor for the sums)."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _model(n, scale, far=0.0):
    """Weakly dispersive random model times scale; `far` shifts its last orbital's energy."""
    m = I.random_hermitian_model(n, 40 + n)
    t = np.where(np.any(m.R != 0, axis=1), 0.03, 1.0) * m.t
    t = np.where((m.i == n - 1) & (m.j == n - 1) & ~np.any(m.R != 0, axis=1), t + far, t)
    return I.HoppingList(n=n, R=m.R, i=m.i, j=m.j, t=scale * t, dim=m.dim)


def _check(lib, ctx, model, plane, p):
    ph, gap = lib.wilson_loop(model, plane, p, precision="fp64", ctx=ctx, gap_tol=0.0)
    ref, rgap = oracle.wilson_loop(model, plane, p, gap_tol=0.0)
    norm = np.bincount(model.i, np.abs(model.t)).max()
    assert np.max(np.abs(gap.cpu().numpy() - rgap)) <= 8 * model.n * EPS * norm
    assert circ_err_rows(ph.cpu().numpy(), ref) <= 1e-10


@pytest.mark.parametrize("scale", [1e-100, 1e-30, 1e-19, 1e20, 1e100])
@pytest.mark.parametrize("n,p", [(4, 2), (12, 5), (40, 20), (66, 13)])
def test_unit_of_energy(lib, ctx, n, p, scale):
    _check(lib, ctx, _model(n, scale), I.Plane(6, 3), p)


@pytest.mark.parametrize("n,p", [(4, 2), (12, 5), (32, 16), (40, 20), (66, 13)])
def test_level_far_from_the_edge(lib, ctx, n, p):
    _check(lib, ctx, _model(n, 1.0, far=1e6), I.Plane(6, 3), p)
