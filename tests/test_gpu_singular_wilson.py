"""Wilson matrices of low rank: pairs of copies of a four-band model exchange their four
occupied states along the loop (their on-site energies swap order), so that the overlaps at
the exchange, and with them half or so of the singular values of the loop matrix, vanish up
to a weak coupling.  The eigenphase solvers must converge, and the phases of the copies that
do not take part stay those of the copy alone.

The coupling E (random, |E| <= 2 sqrt(n) eps) moves those phases by at most about
N |E| / gap = 16 x 2 sqrt(288) x 1e-10 = 5e-8 rad (gap >= 1); the bound asked is 1e-6."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu
N, ROWS, EPS = 16, 6, 1e-10


def exchange_model(stable, pairs, eps=EPS, seed=5):
    """`stable` copies that keep their states, `pairs` pairs that exchange them twice a loop;
    the model and the stable copies."""
    rng = np.random.default_rng(seed)
    parts = [I.bbh(rng.uniform(0.4, 0.6), rng.uniform(0.4, 0.6)) if c % 2 else I.bhz_eq7(rng.uniform(1.3, 1.5))
             for c in range(stable + 2 * pairs)]
    m = I.direct_sum(parts)
    n = m.n
    R, i, j, t = [m.R], [m.i], [m.j], [m.t]
    for q in range(2 * pairs):  # +- 20 cos(2 pi kx) on every orbital of the copy
        o = np.arange(4 * (stable + q), 4 * (stable + q) + 4)
        for dx in (1, -1):
            R.append(np.tile(np.array([[dx, 0, 0]], np.int32), (4, 1)))
            i.append(o)
            j.append(o)
            t.append(np.full(4, 10.0 if q % 2 else -10.0, complex))
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    ii, jj = np.nonzero(np.ones((n, n)))
    R.append(np.zeros((n * n, 3), np.int32))
    i.append(ii)
    j.append(jj)
    t.append((eps * 0.5 * (A + A.conj().T))[ii, jj])
    return I.HoppingList(n=n, R=np.concatenate(R), i=np.concatenate(i), j=np.concatenate(j),
                         t=np.concatenate(t), dim=2), parts[:stable]


# p = 12 and 32: one CTA per loop in shared memory; 48 ... 144: the batched loops and the
# solvers of large Wilson matrices (FP64 and double-float)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("stable,pairs", [(2, 2), (8, 4), (8, 8), (12, 10), (16, 12), (24, 24)])
def test_loop_of_low_rank(lib, ctx, stable, pairs, precision):
    model, copies = exchange_model(stable, pairs)
    origin = (0.5 / N, 0.021, 0.0)  # cos(2 pi kx) away from zero: no closed gap on the grid
    ph, _ = lib.wilson_loop(model, I.Plane(N, ROWS, origin=origin), model.n // 2, precision=precision,
                            ctx=ctx, gap_tol=0.0)  # raises ENOCONV when a solver gives up
    ph = ph.cpu().numpy()
    assert np.all(np.isfinite(ph))
    for r in range(ROWS):
        row = I.Plane(N, 1, origin=(origin[0], origin[1] + r / ROWS, 0.0))
        for c in copies:
            for x in oracle.wilson_loop(c, row, 2, gap_tol=0.0)[0][0]:
                assert np.min(np.abs(np.angle(np.exp(1j * (ph[r] - x))))) <= 1e-6
