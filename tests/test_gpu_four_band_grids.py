"""Four-band models on large grids: one thread per k-point where H(k) ends after a few Jacobi
rotations, four lanes otherwise.  Every row of a large grid against the same rows as small
grids (which take the four-lane kernel, FP64 states to rounding: 1e-10 on phases, 1e-12 on gaps
and projected spin values of order one), and sampled rows, the last CTA's partial one
among them, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu
N, NT, PART = 11, 1301, 1000  # 14 311 points; at most 11 000 in a part
SZ = I.SPIN_HALL_SZ


def blocks(seed, offset=0.0):
    """Two independent random 2 x 2 blocks, orbitals (0, 2) and (1, 3), over 15 translations: with
    a spin operator a plan too long for the launch parameter.  With an offset of the second
    block's energy no level of one block crosses one of the other, so that every p has a gap
    and the occupied states do not jump between the blocks along a loop."""
    rng = np.random.default_rng(seed)
    half = [(1, 0), (0, 1), (1, 1), (1, -1), (2, 0), (0, 2), (2, 1)]
    R, i, j, t = [], [], [], []
    for x, y in half:
        for b in (0, 1):
            for r in (b, b + 2):
                for c in (b, b + 2):
                    z = 0.08 * (rng.standard_normal() + 1j * rng.standard_normal())
                    R += [(x, y, 0), (-x, -y, 0)]
                    i += [r, c]
                    j += [c, r]
                    t += [z, z.conjugate()]
    for r in (1, 3):
        R.append((0, 0, 0))
        i.append(r)
        j.append(r)
        t.append(offset)
    m = I.spin_hall(0.8)
    return I.HoppingList(n=4, R=np.concatenate([m.R, np.array(R, np.int32)]), i=np.concatenate([m.i, i]),
                         j=np.concatenate([m.j, j]), t=np.concatenate([m.t, t]), dim=2)


MODELS = {"bbh": lambda: I.bbh(0.45, 0.55), "spin_hall": lambda: I.spin_hall(0.9),
          "eq9": lambda: I.choti_eq9(1.0, -1.5), "blocks": lambda: blocks(4), "apart": lambda: blocks(4, 10.0)}


def _parts(origin):
    for i0 in range(0, NT, PART):
        m = min(PART, NT - i0)
        yield i0, m, I.Plane(N, m, origin=(origin[0], origin[1] + i0 / NT, origin[2]),
                             trans_dir=(0.0, m / NT, 0.0))


@pytest.mark.parametrize("name,p", [("bbh", 2), ("spin_hall", 2), ("eq9", 2), ("blocks", 2), ("blocks", 4),
                                    ("apart", 1), ("apart", 2), ("apart", 3)])
def test_large_grid_row_by_row(lib, ctx, name, p):
    model, origin = MODELS[name](), (0.013, 0.037, 0.21)
    plane = I.Plane(N, NT, origin=origin)
    kw = dict(precision="fp64", ctx=ctx)
    ph, gap = (x.cpu().numpy() for x in lib.wilson_loop(model, plane, p, **kw))
    for i0, m, part in _parts(origin):
        sph, sgap = (x.cpu().numpy() for x in lib.wilson_loop(model, part, p, **kw))
        assert circ_err_rows(ph[i0:i0 + m], sph) <= 1e-10
        if p < 4:
            assert np.max(np.abs(gap[i0:i0 + m] - sgap)) <= 1e-12
    for r in (0, 1, 650, NT - 2, NT - 1):
        row = I.Plane(N, 1, origin=(origin[0], origin[1] + r / NT, origin[2]))
        ref, rgap = oracle.wilson_loop(model, row, p)
        if p < 4:
            assert abs(gap[r] - rgap[0]) <= 1e-12
        assert oracle.circular_match_error(ph[r], ref[0]) <= 1e-10


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("name", ["spin_hall", "blocks"])
def test_large_grid_spin_resolved(lib, ctx, name, sign):
    model, origin = MODELS[name](), (0.013, 0.037, 0.0)
    kw = dict(precision="fp64", ctx=ctx)
    big = [x.cpu().numpy() for x in
           lib.spin_resolved_wilson_loop(model, I.Plane(N, NT, origin=origin), 2, SZ, sign, **kw)]
    for i0, m, part in _parts(origin):
        small = [x.cpu().numpy() for x in lib.spin_resolved_wilson_loop(model, part, 2, SZ, sign, **kw)]
        assert circ_err_rows(big[0][i0:i0 + m], small[0]) <= 1e-10
        for a, b in zip(big[1:], small[1:]):
            assert np.max(np.abs(a[i0:i0 + m] - b)) <= 1e-12
    for r in (0, 650, NT - 1):
        row = I.Plane(N, 1, origin=(origin[0], origin[1] + r / NT, 0.0))
        ref = oracle.spin_resolved_wilson_loop(model, row, 2, SZ, sign)
        assert oracle.circular_match_error(big[0][r], ref[0][0]) <= 1e-10
        assert np.max(np.abs(big[1][r] - ref[1][0])) <= 1e-12
