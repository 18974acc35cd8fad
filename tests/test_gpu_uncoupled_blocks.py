"""FP64 requests on models that fall apart into uncoupled blocks (5 <= n <= 32): the hopping list
tells the blocks, and where their Jacobi rotations are few the FP64 solve runs without the FP32 one.

The tolerance is rounding: 8 sqrt(N p) 2^-52 times ten for the eigenvalue conditions of coarse
loops, and gaps to n units 2^-52 of the largest amplitude sum."""
import numpy as np
import pytest

import oracle
from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import circ_err_rows, ctx, lib  # noqa: F401

pytestmark = pytest.mark.gpu


def shuffled(m, seed):
    """The model with its orbitals renumbered, so that the blocks interleave."""
    to = np.random.default_rng(seed).permutation(m.n).astype(np.int32)
    return I.HoppingList(n=m.n, R=m.R, i=to[m.i], j=to[m.j], t=m.t, dim=m.dim)


def with_free_levels(m, energies):
    """The model and isolated orbitals behind it."""
    k, n = len(energies), m.n
    at = np.arange(n, n + k, dtype=np.int32)
    return I.HoppingList(n=n + k, R=np.concatenate([m.R, np.zeros((k, 3), np.int32)]),
                         i=np.concatenate([m.i, at]), j=np.concatenate([m.j, at]),
                         t=np.concatenate([m.t, np.asarray(energies, complex)]), dim=m.dim)


CASES = {
    # few rotations: no FP32 solve
    "two_bbh": (I.direct_sum([I.bbh()] * 2), 4),
    "eight_bbh": (shuffled(I.direct_sum([I.bbh(0.4 + 0.02 * c, 0.5) for c in range(8)]), 1), 16),
    "five_spin_hall": (shuffled(I.direct_sum([I.spin_hall(0.8 + 0.1 * c) for c in range(5)]), 2), 10),
    "free_levels": (shuffled(with_free_levels(I.direct_sum([I.bbh(), I.spin_hall()]), [-4.5, 4.5, 5.0]), 3), 5),
    # many rotations: the FP32 start
    "two_dense_halves": (shuffled(I.direct_sum([I.random_hermitian_model(8, 3)] * 2), 4), 8),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("N,Nt", [(6, 5), (16, 40)])
def test_uncoupled_blocks(lib, ctx, name, N, Nt):
    model, p = CASES[name]
    plane = I.Plane(N, Nt, origin=(0.013, 0.021, 0.0))
    ph, gap = lib.wilson_loop(model, plane, p, precision="fp64", gap_tol=0.0, ctx=ctx)
    ref, ref_gap = oracle.wilson_loop(model, plane, p, gap_tol=0.0)
    assert circ_err_rows(ph.cpu().numpy(), ref) <= 80.0 * (N * p) ** 0.5 * 2.0 ** -52
    assert np.abs(gap.cpu().numpy() - ref_gap).max() <= model.n * 2.0 ** -52 * np.abs(model.t).sum()


def test_spin_sector_of_uncoupled_blocks(lib, ctx):
    copies = 3
    model = I.direct_sum([I.spin_hall(0.8 + 0.1 * c) for c in range(copies)])
    spin = np.kron(np.eye(copies), I.SPIN_HALL_SZ)
    plane, p = I.Plane(8, 9, origin=(0.013, 0.021, 0.0)), 2 * copies
    ph = lib.spin_resolved_wilson_loop(model, plane, p, spin, -1, precision="fp64", ctx=ctx)[0]
    ref = oracle.spin_resolved_wilson_loop(model, plane, p, spin, -1)[0]
    assert circ_err_rows(ph.cpu().numpy(), ref) <= 80.0 * (plane.N * copies) ** 0.5 * 2.0 ** -52
