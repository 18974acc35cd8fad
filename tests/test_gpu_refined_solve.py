"""FP64 requests at n <= 32: an FP32 eigenbasis refined to FP64, or the FP64 Jacobi solve
where a band edge leaves the refinement's range.  Phases against the oracle within the
FP64 bound of the other parity tests; gaps within 8 n eps ||H|| (the forward error of a
backward-stable eigenvalue, with a factor for the sums of n terms)."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _check(lib, ctx, model, plane, p, phases=True):
    ph, gap = lib.wilson_loop(model, plane, p, precision="fp64", ctx=ctx, gap_tol=0.0)
    ref, rgap = oracle.wilson_loop(model, plane, p, gap_tol=0.0)
    norm = np.bincount(model.i, np.abs(model.t)).max()  # bounds ||H(k)||
    assert np.max(np.abs(gap.cpu().numpy() - rgap)) <= 8 * model.n * EPS * norm
    if phases:
        assert circ_err_rows(ph.cpu().numpy(), ref) <= 1e-10


def _scaled(m, s, hop=1.0):
    """The model times s, its hoppings between cells times hop as well."""
    t = s * m.t * np.where(np.any(m.R != 0, axis=1), hop, 1.0)
    return I.HoppingList(n=m.n, R=m.R, i=m.i, j=m.j, t=t, dim=m.dim)


@pytest.mark.parametrize("n,p", [(2, 1), (4, 1), (4, 2), (4, 3), (5, 1), (8, 7), (17, 8), (31, 16), (32, 1), (32, 31)])
def test_refined_states_and_gap(lib, ctx, n, p):
    # weak dispersion: the overlaps of neighbouring points stay near one, so that the
    # eigenphases of their product are well conditioned
    _check(lib, ctx, _scaled(I.random_hermitian_model(n, 11 + n), 1.0, hop=0.03), I.Plane(9, 5), p)


@pytest.mark.parametrize("copies", [1, 2, 5])
@pytest.mark.parametrize("split", [0.0, 1e-9, 1e-6, 1e-3])
def test_near_degenerate_band_edges(lib, ctx, copies, split):
    """Copies of the quadrupole insulator whose levels differ by `split`: the occupied and
    the unoccupied edge are clusters of 2 to 10 levels."""
    parts = []
    for c in range(copies):
        m = I.bbh(0.5, 0.5)
        on = I.HoppingList(n=4, R=np.concatenate([m.R, np.zeros((4, 3), np.int32)]),
                           i=np.concatenate([m.i, np.arange(4)]), j=np.concatenate([m.j, np.arange(4)]),
                           t=np.concatenate([m.t, np.full(4, c * split + 0j)]), dim=m.dim)
        parts.append(on)
    model = I.direct_sum(parts) if copies > 1 else parts[0]
    _check(lib, ctx, model, I.Plane(8, 5), 2 * copies)


@pytest.mark.parametrize("n", [4, 12])
@pytest.mark.parametrize("offset", [1e-7, 1e-4, 1e-2])
def test_gap_down_to_closing(lib, ctx, n, offset):
    """Two identical blocks shifted against each other by `offset`: with p = 1 the direct gap
    is the offset itself, on both sides of the refinement's limit."""
    m = I.random_hermitian_model(n // 2, 3)
    k = n // 2
    sh = I.HoppingList(n=k, R=np.concatenate([m.R, np.zeros((k, 3), np.int32)]),
                       i=np.concatenate([m.i, np.arange(k)]), j=np.concatenate([m.j, np.arange(k)]),
                       t=np.concatenate([m.t, np.full(k, offset + 0j)]), dim=m.dim)
    _check(lib, ctx, I.direct_sum([m, sh]), I.Plane(7, 4), 1, phases=False)


@pytest.mark.parametrize("scale", [1e-30, 1e-9, 1e20])
def test_energy_scale_outside_fp32(lib, ctx, scale):
    for n, p in ((4, 2), (10, 4)):
        _check(lib, ctx, _scaled(I.random_hermitian_model(n, 5), scale, hop=0.03), I.Plane(7, 4), p)


# ---- n > 32: the FP32 solve with the FP64 polish, the FP64 solve where it does not apply


@pytest.mark.parametrize("n,p", [(33, 1), (33, 16), (40, 32), (41, 33), (63, 31), (64, 62), (97, 65)])
def test_polished_states_and_gap(lib, ctx, n, p):
    """Dense models: both column tiles (p <= 32 and beyond) and their remainders."""
    _check(lib, ctx, _scaled(I.random_hermitian_model(n, 11 + n), 1.0, hop=0.03), I.Plane(6, 3), p)


@pytest.mark.parametrize("copies", [9, 11])
@pytest.mark.parametrize("split", [0.0, 1e-6, 2e-3])
def test_polished_degenerate_edges(lib, ctx, copies, split):
    """Sparse models whose band edges hold 2 to 22 levels: small clusters in the polish, larger
    ones in the FP64 solve."""
    parts = []
    for c in range(copies):
        m = I.bbh(0.5, 0.5)
        parts.append(I.HoppingList(n=4, R=np.concatenate([m.R, np.zeros((4, 3), np.int32)]),
                                   i=np.concatenate([m.i, np.arange(4)]), j=np.concatenate([m.j, np.arange(4)]),
                                   t=np.concatenate([m.t, np.full(4, c * split * c + 0j)]), dim=m.dim))
    _check(lib, ctx, I.direct_sum(parts), I.Plane(6, 3), 2 * copies)


@pytest.mark.parametrize("offset", [1e-7, 1e-4, 1e-2])
def test_polished_gap_down_to_closing(lib, ctx, offset):
    m = I.random_hermitian_model(20, 3)
    sh = I.HoppingList(n=20, R=np.concatenate([m.R, np.zeros((20, 3), np.int32)]),
                       i=np.concatenate([m.i, np.arange(20)]), j=np.concatenate([m.j, np.arange(20)]),
                       t=np.concatenate([m.t, np.full(20, offset + 0j)]), dim=m.dim)
    _check(lib, ctx, I.direct_sum([m, sh]), I.Plane(6, 3), 1, phases=False)


def test_polish_without_room_takes_the_fp64_solve(lib):
    """A budget that holds the FP64 solve's slot (0.6 MiB) but not the polish's (1.6 MiB)."""
    model = I.direct_sum([_scaled(I.random_hermitian_model(4, 5 + b), 1.0, hop=0.03) for b in range(50)])
    small = lib.Context(0, mem_budget_bytes=5 << 18)
    try:
        _check(lib, small, model, I.Plane(3, 1), 1, phases=False)
    finally:
        small.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_spin_split_of_two_bands_at_large_n(lib, ctx, precision):
    """n = 36, p = 2: the projected spin operator is 2 x 2, the smallest matrix of the
    tridiagonal eigensolver.  Two spin blocks, one shifted by less than the gap."""
    m = _scaled(I.random_hermitian_model(18, 8), 1.0, hop=0.03)
    up = I.HoppingList(n=18, R=np.concatenate([m.R, np.zeros((18, 3), np.int32)]),
                       i=np.concatenate([m.i, np.arange(18)]), j=np.concatenate([m.j, np.arange(18)]),
                       t=np.concatenate([m.t, np.full(18, 0.02 + 0j)]), dim=m.dim)
    model, S = I.direct_sum([m, up]), np.diag(np.repeat([1.0, -1.0], 18))
    plane = I.Plane(6, 3)
    ref, rpso, _, _ = oracle.spin_resolved_wilson_loop(model, plane, 2, S, -1)
    ph, pso, _, _ = lib.spin_resolved_wilson_loop(model, plane, 2, S, -1, precision=precision, ctx=ctx)
    assert circ_err_rows(ph.cpu().numpy(), ref) <= (1e-10 if precision == "fp64" else 1e-6)
    assert np.abs(pso.cpu().numpy() - rpso).max() <= 1e-9


@pytest.mark.parametrize("p", [1, 2, 3])
def test_sparse_four_band_model_on_a_large_grid(lib, ctx, p):
    """n = 4 with entries that are identically zero, past 8192 k-points: one thread per k-point;
    row 0 against the oracle and the small grid of the same row against the large one."""
    t = I.bbh(0.5, 0.7)
    on = I.HoppingList(n=4, R=np.concatenate([t.R, np.zeros((4, 3), np.int32)]), i=np.concatenate([t.i, np.arange(4)]),
                       j=np.concatenate([t.j, np.arange(4)]),
                       t=np.concatenate([t.t, np.array([0.0, 0.3, 0.7, 1.1]) + 0j]), dim=t.dim)
    ph, gap = lib.wilson_loop(on, I.Plane(11, 751), p, precision="fp64", ctx=ctx, gap_tol=0.0)
    ref, rgap = oracle.wilson_loop(on, I.Plane(11, 1), p, gap_tol=0.0)
    assert abs(float(gap[0]) - rgap[0]) <= 8 * 4 * EPS * 4.0
    assert circ_err_rows(ph[:1].cpu().numpy(), ref) <= 1e-10
